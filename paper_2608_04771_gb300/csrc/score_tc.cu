// score_tc.cu -- tensor-core (tcgen05) passes of the Eq. 2 cache scores for bf16 caches.
//
// Both passes are persistent (one CTA per SM walking an equal contiguous range of the call's
// work, planned from the lengths by every CTA itself, barrier phases running on across units):
//   warp 0  : TMA producer (window queries once per unit, then a ring of K tiles of 128 keys)
//   warp 1  : allocates 512 TMEM columns, issues tcgen05.mma (bf16 in, fp32 accumulate in
//             TMEM) and commits to mbarriers
//   warps 2..: epilogue groups of four warps, reading accumulators with tcgen05.ld (one TMEM
//             lane per thread) into the softmax arithmetic
// Operands sit in shared memory in the 128-byte-swizzled K-major layout the TMA writes
// (rows of 64 bf16, 8-row atoms of 1024 bytes); each MMA takes a K=16 slice.  The
// accumulators rotate through a ring of TMEM regions, so the MMAs of the next tiles run
// while the epilogue groups work on earlier ones.
//
// Pass 1 (row statistics): queries on M (128-row tiles), keys on N, so each thread owns
//   one window row and keeps a (reference, sum) over the chunk's keys.
// Pass 2 (column sums): keys on M (128 per tile), queries on N, so each thread sums
//   2^(c*l - b_r) over a range of the window rows for one key.
//
// What bounds both: HBM, from which each pass reads all keys (two thirds of the 7B-class call below are
// the time of its 3.6 GB of keys, read twice, at the copy rate); the epilogue's instruction issue, about 3.3 instructions per
// exponential (scale and subtract, exponential, add, a share of the loads) where the special-function
// unit takes one per four cycles; and the MMA issuer's waits between tiles.  Whole calls replayed from a
// graph, us, on the 7B-class heads (28 x 8 x 4 units, 224 window rows, 15000 to 16384 keys; both passes,
// combine and pool) and in one pass over 8 layers of the 32B-class heads (320 rows, 32768 keys):
//   before (every epilogue warp on every tile, sizes tested per 8 columns)      1800        900
//   now (see the comments at the plan, the groups and the batches)              1540-1570   620-630
//   (as calls among others 1610-1625 and 640)
// Every mbarrier wait is bounded; a wait that runs out sets the device error word and
// the CTA stops issuing work, waits (bounded) for nothing further and frees its TMEM.
#include <cuda.h>

#include "common.cuh"
#include "internal.h"
#include "score_plan.cuh"
#include "tma.cuh"

namespace reco {

// ---------------------------------------------------------------- tcgen05 wrappers
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]^T, kind::f16 (both operands bf16 here).
__device__ __forceinline__ void tc_mma(uint32_t dtmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(dtmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// TMEM loads into registers do not wait: tmem_ld_wait_regs() comes before their use.
// 8 consecutive fp32 columns of the calling thread's TMEM lane (no wait).
__device__ __forceinline__ void tmem_ld8_nowait(uint32_t taddr, float *v)
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 consecutive fp32 columns of the calling thread's TMEM lane (no wait).
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, float *v)
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Wait for this thread's TMEM loads, then pass the NV loaded registers through an empty
// asm so that no use of them can be scheduled before the wait.
template <int NV>
__device__ __forceinline__ void tmem_ld_wait_regs(float *v)
{
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < NV; i += 8)
        asm volatile(""
                     : "+f"(v[i]), "+f"(v[i + 1]), "+f"(v[i + 2]), "+f"(v[i + 3]), "+f"(v[i + 4]), "+f"(v[i + 5]),
                       "+f"(v[i + 6]), "+f"(v[i + 7]));
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row atoms of
// 1024 bytes (stride byte offset 1024), descriptor version 1.  The start address sits in
// the low 14 bits as address / 16; a shared-memory address stays below 2^18 bytes, so
// the descriptor of (address + offset) is this one plus offset / 16 (no carry out).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)1u << 16;            // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024u >> 4) << 32;  // stride byte offset
    d |= (uint64_t)1u << 46;            // version
    d |= (uint64_t)2u << 61;            // SWIZZLE_128B
    return d;
}

// Instruction descriptor, kind::f16: bf16 A and B (K-major), fp32 D, shape M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

constexpr long long kTcSpin = 1LL << 22;  // polls, each suspended for up to a few microseconds
constexpr int kTcMaxR = 512;  // window rows (G*w) the tensor-core passes take
constexpr int kTmemCols = 512;

// Bounded wait of a converged warp on an mbarrier phase; the same answer in every lane.  A wait
// that runs out raises the CTA's abort flag, which ends the other roles' waits too.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, unsigned *err)
{
    for (long long i = 0; i < kTcSpin; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if ((i & 1023) == 1023 && __any_sync(0xffffffffu, *abort_flag != 0)) return false;
    }
    *abort_flag = 1;
    raise_error(err, ERR_INTERNAL);
    return false;
}

// Whether an mbarrier phase has completed, without waiting (a converged warp).
__device__ __forceinline__ bool warp_test(uint32_t bar, uint32_t parity)
{
    return __all_sync(0xffffffffu, mbar_test(bar, parity));
}

// TMEM columns between pass-2 accumulator buffers: a block's width rounded up to 32.
__host__ __device__ constexpr int p2_stride(int cb) { return (cb + 31) & ~31; }

// Split n columns (a multiple of 8) into `parts` contiguous ranges of multiples of 8.
__device__ __forceinline__ int split8_lo(int n, int parts, int g) { return ((n / 8) * g / parts) * 8; }

// One lane of a converged warp (elect.sync, so that the compiler knows that a single thread
// runs the block it guards: tcgen05 and TMA instructions take their operands from uniform
// registers, and a `lane == 0` guard made it fill them the slow way).
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}" : "=r"(p));
    return p != 0;
}

// ---------------------------------------------------------------- pass 1: row statistics
// A piece is the accumulator of one 128-row query tile mt against one tile of 128 keys; the
// pieces p = gt * MT + mt rotate through four TMEM regions of 128 columns.  A group of four
// epilogue warps takes query tile mt of every EG-th key tile, whole: the groups work on
// different regions and so drift apart, one exponentiating while another waits for its
// accumulator, and a region is released by four warps.  Where a unit has few tiles (SPLIT, for
// caches of at most kSplitCap rows) that leaves groups idle and a tile's columns to one of them:
// there every group takes its share of every tile's columns (4 units of 120 keys, both passes, 15.2 -> 14.2 us,
// 160 of 500 keys 31.8 -> 30.4; 16384 keys 1.57 -> 1.61 ms).
constexpr int kSplitCap = 1024;
template <int D, int MT, int EG, bool SPLIT>
struct Pass1Cfg {
    static constexpr int CW = SPLIT ? kTile / EG : kTile;  // columns of a piece that a group takes
    static constexpr int HALVES = D / 64;
    static constexpr int BOX = kTile * 128;  // 128 rows x 128 bytes
    static constexpr int KSTAGE = HALVES * BOX;
    static constexpr int NR = kTmemCols / kTile;  // TMEM regions
    static constexpr int QBYTES = MT * HALVES * BOX;
    static constexpr int NS0 = (200 * 1024 - QBYTES) / KSTAGE;
    static constexpr int NS = NS0 > 8 ? 8 : NS0;
    static constexpr size_t SMEM = 1024 + (size_t)QBYTES + (size_t)NS * KSTAGE;
    static constexpr int THREADS = 64 + 128 * MT * EG;
    static_assert((NR & (NR - 1)) == 0 && NR >= MT, "accumulator ring");
    static_assert((EG & (EG - 1)) == 0, "tiles are dealt by their low bits");
    static_assert(NS >= 2, "K ring too short");
    static_assert(THREADS <= 576, "96 registers a thread");
};

// Exponent of a normal positive float, as an integer power of two.
__device__ __forceinline__ int exp2_of(float z) { return ((__float_as_int(z) >> 23) & 0xff) - 127; }

// One row's running (reference m, sum z) over 16 accumulator columns v (logit = v * c2 in log2
// units), of which columns 0..lim are visible, with their max taken first.
__device__ __forceinline__ void rowstats_exact(const float (&v)[16], int lim, float c2, float &m, float &z)
{
    float mx = -INFINITY;
#pragma unroll
    for (int q = 0; q < 16; ++q)
        if (q <= lim) mx = fmaxf(mx, v[q]);
    const float mn = fmaxf(m, mx * c2);
    if (mn == -INFINITY) return;
    const float nb = -mn;
    float a4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int q = 0; q < 16; ++q) a4[q & 3] += q <= lim ? fast_exp2(fmaf(v[q], c2, nb)) : 0.f;
    z = z * fast_exp2(m - mn) + ((a4[0] + a4[1]) + (a4[2] + a4[3]));
    m = mn;
}

// Largest of the 16 columns at ta.
__device__ __forceinline__ float rowmax16(uint32_t ta)
{
    float v[16];
    tmem_ld16_nowait(ta, v);
    tmem_ld_wait_regs<16>(v);
    float mx = v[0];
#pragma unroll
    for (int q = 1; q < 16; ++q) mx = fmaxf(mx, v[q]);
    return mx;
}

// Sum over the N columns at ta of 2^(v * c2 - m), two TMEM loads in flight.
template <int N> __device__ __forceinline__ float rowsum_tile(uint32_t ta, float c2, float m)
{
    const float nb = -m;
    float v[2][16], a4[4] = {0.f, 0.f, 0.f, 0.f};
    tmem_ld16_nowait(ta, v[0]);
#pragma unroll
    for (int k = 0; k < N / 16; ++k) {
        tmem_ld_wait_regs<16>(v[k & 1]);
        if (k + 1 < N / 16) tmem_ld16_nowait(ta + 16 * (k + 1), v[(k + 1) & 1]);
#pragma unroll
        for (int q = 0; q < 16; ++q) a4[q & 3] += fast_exp2(fmaf(v[k & 1][q], c2, nb));
    }
    return (a4[0] + a4[1]) + (a4[2] + a4[3]);
}

template <int D, int MT, int EG, bool SPLIT>
__global__ void __launch_bounds__(Pass1Cfg<D, MT, EG, SPLIT>::THREADS, 1)
    score_rowstats_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                      const int32_t *__restrict__ lens, ScoreMask mask, int w, int G, int Hq, int Hkv, int L_cap, int R,
                      int n_chunks, int units, float c2, float *__restrict__ part_m, float *__restrict__ part_z,
                      unsigned *err)
{
    using C = Pass1Cfg<D, MT, EG, SPLIT>;
    constexpr int HALVES = C::HALVES, BOX = C::BOX, KSTAGE = C::KSTAGE;
    constexpr int NR = C::NR, NS = C::NS, N = kTile, CW = C::CW;
    constexpr int CT = kScoreChunk / kTile;  // tiles per chunk
    constexpr uint32_t IDESC = idesc_bf16(128, N);
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar_qfull, bar_qempty, bar_kfull[NS], bar_kempty[NS], bar_afull[NR],
        bar_aempty[NR];
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh;
    __shared__ TilePlan plan;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t raw0 = smem_addr(smem_raw);
    const uint32_t base = (raw0 + 1023u) & ~1023u;
    const uint32_t Qs = base;              // MT x HALVES x BOX
    const uint32_t Ks = base + C::QBYTES;  // NS x KSTAGE
    if (tid == 0) {
        prefetch_tensormap(&tmQ);
        prefetch_tensormap(&tmK);
        mbar_init(smem_addr(&bar_qfull), 1);
        mbar_init(smem_addr(&bar_qempty), 1);
        for (int s = 0; s < NS; ++s) {
            mbar_init(smem_addr(&bar_kfull[s]), 1);
            mbar_init(smem_addr(&bar_kempty[s]), 1);
        }
        for (int b = 0; b < NR; ++b) {
            mbar_init(smem_addr(&bar_afull[b]), 1);
            mbar_init(smem_addr(&bar_aempty[b]), SPLIT ? 4 * EG : 4);
        }
        abort_sh = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_shared();
    }
    if (warp == 1) {
        tmem_alloc(smem_addr(&tmem_sh), kTmemCols);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    volatile int *abort_flag = &abort_sh;
    // everything above runs while the previous kernel drains; from here on its outputs
    // (lens, the window queries) are read
    wait_prior_grid();

    bool ok = true;
    int gt = 0, nq = 0;  // tiles and query loads so far (each role counts its own)
    bool a_ready = false, k_ready = false;  // MMA issuer: the next piece's region, the next tile's keys
    for (int skip = 0, n_runs = 1; skip < n_runs; skip += kPlanRuns) {
        n_runs = plan_runs_call(plan, lens, mask, w, L_cap, units, false, kScoreChunk, skip, nullptr, nullptr, err);
        const int n_here = min(kPlanRuns, n_runs - skip);
        if (warp == 0) {  // producer: a unit's window queries, then its run's K tiles
            for (int e = 0; ok && e < n_here; ++e) {
                const TileRun run = plan.run[e];
                if (nq > 0 && !(ok = warp_wait(smem_addr(&bar_qempty), (nq - 1) & 1, abort_flag, err))) break;
                if (elect_one()) {
                    const long lb = run.u / Hkv;
                    const int q_row0 = (int)((lb * Hq + (run.u % Hkv) * G) * w);
                    mbar_expect_tx(smem_addr(&bar_qfull), (uint32_t)C::QBYTES);
                    for (int mt = 0; mt < MT; ++mt)
                        for (int hh = 0; hh < HALVES; ++hh)
                            tma_load_2d(Qs + (mt * HALVES + hh) * BOX, &tmQ, 64 * hh, q_row0 + 128 * mt,
                                        smem_addr(&bar_qfull));
                }
                ++nq;
                const int k_row0 = run.u * L_cap + run.t0 * N;
                for (int t = 0; t < run.nt; ++t, ++gt) {
                    const int s = gt % NS;
                    if (!(ok = warp_wait(smem_addr(&bar_kempty[s]), ((gt / NS) & 1) ^ 1, abort_flag, err))) break;
                    if (elect_one()) {
                        mbar_expect_tx(smem_addr(&bar_kfull[s]), KSTAGE);
                        for (int hh = 0; hh < HALVES; ++hh)
                            tma_load_2d(Ks + s * KSTAGE + hh * BOX, &tmK, 64 * hh, k_row0 + t * N,
                                        smem_addr(&bar_kfull[s]));
                    }
                }
            }
        } else if (warp == 1) {  // MMA issuer
            for (int e = 0; ok && e < n_here; ++e) {
                const int nt = plan.run[e].nt;
                if (!(ok = warp_wait(smem_addr(&bar_qfull), nq & 1, abort_flag, err))) break;
                ++nq;
                for (int t = 0; ok && t < nt; ++t, ++gt) {
                    const int s = gt % NS;
                    if (!k_ready && !(ok = warp_wait(smem_addr(&bar_kfull[s]), (gt / NS) & 1, abort_flag, err))) break;
#pragma unroll
                    for (int mt = 0; mt < MT; ++mt) {
                        const int p = gt * MT + mt, b = p % NR;
                        if (!a_ready &&
                            !(ok = warp_wait(smem_addr(&bar_aempty[b]), ((p / NR) & 1) ^ 1, abort_flag, err)))
                            break;
                        tc_fence_after();
                        // descriptors of the first K slice; later slices add their offset / 16
                        const uint32_t d = tmem + (uint32_t)(b * N);
                        const uint64_t ad0 = sw128_desc(Qs + mt * HALVES * BOX);
                        const uint64_t bd0 = sw128_desc(Ks + s * KSTAGE);
                        auto issue = [&](int k) {
                            const uint64_t off = (uint64_t)(((k >> 2) * BOX + (k & 3) * 32) >> 4);
                            tc_mma(d, ad0 + off, bd0 + off, IDESC, k > 0 ? 1u : 0u);
                        };
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < D / 32; ++k) issue(k);
                        }
                        __syncwarp();
                        {  // the next piece's barriers, looked at while these MMAs run
                            const int b1 = (p + 1) % NR, s1 = (gt + 1) % NS;
                            a_ready = warp_test(smem_addr(&bar_aempty[b1]), (((p + 1) / NR) & 1) ^ 1);
                            if (mt == MT - 1) k_ready = warp_test(smem_addr(&bar_kfull[s1]), ((gt + 1) / NS) & 1);
                        }
                        if (elect_one()) {
#pragma unroll
                            for (int k = D / 32; k < D / 16; ++k) issue(k);
                            tc_commit(smem_addr(&bar_afull[b]));
                            if (mt == MT - 1) {
                                tc_commit(smem_addr(&bar_kempty[s]));
                                if (t == nt - 1) tc_commit(smem_addr(&bar_qempty));  // queries free once these land
                            }
                        }
                        __syncwarp();
                    }
                }
            }
        } else {  // epilogue: query tile mt of every EG-th key tile (or CW columns of all), one window row per thread
            const int idx = (warp - 2) >> 2, mt = idx / EG, g = idx % EG, quarter = warp & 3;
            const int r = mt * 128 + quarter * 32 + lane;
            const bool warp_rows = mt * 128 + quarter * 32 < R;  // this warp holds real window rows
            const int t_row = r % w;
            for (int e = 0; ok && e < n_here; ++e) {
                const TileRun run = plan.run[e];
                const int jmax = run.L - w + t_row;  // last key this window row sees
                const int t_end = run.t0 + run.nt;
                for (int c0 = run.t0; ok && c0 < t_end; c0 += CT) {  // chunk by chunk: one partial each
                    const int c1 = min(c0 + CT, t_end);
                    const int j1 = min(c1 * N, run.L);
                    // this group's tiles: every EG-th of the CTA's, so that it always meets its own TMEM
                    // regions.  They are every EG-th of the chunk's from its tile `first`: the partial goes
                    // by that, so a unit's partials do not depend on the plan
                    const int first = SPLIT ? g : (g - gt) & (EG - 1), t0 = SPLIT ? c0 : c0 + first;
                    const int col = SPLIT ? g * CW : 0;
                    float m = -INFINITY, z = 0.f;  // reference (log2 units) and sum relative to it
                    for (int t = t0; t < c1; t += SPLIT ? 1 : EG) {
                        const int p = (gt + t - c0) * MT + mt, b = p % NR;
                        if (!(ok = warp_wait(smem_addr(&bar_afull[b]), (p / NR) & 1, abort_flag, err))) break;
                        tc_fence_after();
                        if (warp_rows) {
                            const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * N + col);
                            const int lim = min(j1 - 1, jmax) - t * N - col;  // columns 0..lim are visible
                            // a tile that every row sees whole is summed against the rows' references (at
                            // first the max of 16 columns) with no max pass; a masked tile, or a sum that
                            // could overflow (or is NaN), takes the rows' maxima, 16 columns at a time
                            bool summed = false;
                            if (__all_sync(0xffffffffu, lim >= CW - 1)) {
                                if (t == t0) m = rowmax16(ta) * c2;
                                if (__all_sync(0xffffffffu, m > -INFINITY)) {
                                    const float sum = rowsum_tile<CW>(ta, c2, m);
                                    summed = __all_sync(0xffffffffu, sum <= 0x1p96f);
                                    if (summed) z += sum;
                                }
                                if (!summed && t == t0) m = -INFINITY;
                            }
                            if (!summed) {
#pragma unroll 1
                                for (int k = 0; k < CW / 16; ++k) {
                                    float v[16];
                                    tmem_ld16_nowait(ta + 16 * k, v);
                                    tmem_ld_wait_regs<16>(v);
                                    if (lim >= 16 * k) rowstats_exact(v, lim - 16 * k, c2, m, z);
                                }
                            }
                            if (z > 0x1p64f) {  // move the reference up by a power of two: exact rescale
                                const int k = exp2_of(z);
                                z = __int_as_float(__float_as_int(z) - (k << 23));
                                m += (float)k;
                            }
                        }
                        tc_fence_before();  // every column of the piece read: release the region
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_addr(&bar_aempty[b]));
                    }
                    gt += c1 - c0;
                    if (ok && r < R) {
                        const size_t o = (((size_t)run.u * n_chunks + c0 / CT) * EG + first) * R + r;
                        part_m[o] = m;
                        part_z[o] = z;
                    }
                }
            }
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ---------------------------------------------------------------- pass 2: column sums
// The NQ query columns of a key tile are one MMA chain (NP = 1, NW = NQ <= 256) or two
// (NP = 2, NW = NQ / 2); each chain's accumulator is a piece in a ring of NR TMEM regions.
// The four groups of four epilogue warps are two sets that take the key tiles in turn, the groups
// of a set splitting each piece's columns, one key per thread: the sets drift apart, so that one
// exponentiates while the other waits.  A set must not meet a region whose piece before its own
// may still be the other set's (the barrier's parity could not tell the two): with two chains and
// only two regions (NQ > 320) all groups form one set.  So they do where every tile has a CTA of its
// own (no second tile to drift to).
// SHORT: calls of at most kShortTiles tiles per CTA, which a few us of planning would stretch, have the
// plan inline and their barriers set by a warp: the trace's boundary takes 16.8 us, 19.1 otherwise;
// its cache of 1024 rows 23.2 and 25.0; 1792 units of 500 to 960
// keys, all scored, take the same either way, long calls 1 to 2% less without.
constexpr int kShortTiles = 128;
constexpr int kP2Groups = 4;
constexpr int kP2Slots = 4;  // tiles whose other ranges' sums may wait for the first range's warps

// The log2 normalisers of N columns (16-byte aligned shared memory; +inf for padding).
template <int N> __device__ __forceinline__ void colsum_norms(const float *b, float (&nb)[16])
{
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
        const float4 x = *reinterpret_cast<const float4 *>(b + 4 * i);
        nb[4 * i] = x.x;
        nb[4 * i + 1] = x.y;
        nb[4 * i + 2] = x.z;
        nb[4 * i + 3] = x.w;
    }
}

// a4 += sum over N columns of 2^(v * c2 - b).
template <int N>
__device__ __forceinline__ void colsum_batch(const float (&v)[16], const float (&nb)[16], float c2, float (&a4)[4])
{
#pragma unroll
    for (int i = 0; i < N; ++i) a4[i & 3] += fast_exp2(fmaf(v[i], c2, -nb[i]));
}

// One step of a piece: the 16 columns in `cur` (their load is in flight) while the next 16 (or the
// last 8) load into `nxt`.  Returns false after the range's last columns.
template <typename Release>
__device__ __forceinline__ bool colsum_step(uint32_t &ta, const float *&b, int &left, float (&cur)[16],
                                            float (&nxt)[16], float c2, float (&a4)[4], Release release)
{
    float bb[16];
    colsum_norms<16>(b, bb);  // read before the wait for the accumulator columns
    tmem_ld_wait_regs<16>(cur);
    left -= 16;
    ta += 16;
    b += 16;
    if (left >= 16) tmem_ld16_nowait(ta, nxt);
    else if (left == 8) tmem_ld8_nowait(ta, nxt);
    else release();
    colsum_batch<16>(cur, bb, c2, a4);
    if (left >= 16) return true;
    if (left == 8) {
        colsum_norms<8>(b, bb);
        tmem_ld_wait_regs<8>(nxt);
        release();
        colsum_batch<8>(nxt, bb, c2, a4);
    }
    return false;
}

template <int D, bool SHORT>
__global__ void __launch_bounds__(64 + 128 * kP2Groups, 1)
    score_colsum_tc(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const int32_t *__restrict__ lens, ScoreMask mask, int w, int G, int Hq, int Hkv, int L_cap, int R,
                    int NQ, int NP, int NR, int NS, int sets, int units, float c2, const float *__restrict__ rowb,
                    const float *__restrict__ row_lse, long rows_q, float *__restrict__ raw, int32_t *ulist,
                    int32_t *ucount, unsigned *err)
{
    constexpr int HALVES = D / 64;
    constexpr int KBOX = kTile * 128;  // 128 keys x 128 bytes
    constexpr int KSTAGE = HALVES * KBOX;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar_qfull, bar_qempty, bar_kfull[4], bar_kempty[4], bar_afull[4], bar_aempty[4],
        bar_part[8][kP2Slots];
    __shared__ float part_sh[48][32];  // [(set, quarter)][slot][ranges after the first]
    __shared__ uint32_t tmem_sh;
    __shared__ int abort_sh;
    __shared__ TilePlan plan;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int split = kP2Groups / sets;  // column ranges of a piece (two or four)
    const int NW = NQ / NP;              // columns of one piece
    const int stride = (NW + 31) & ~31;  // TMEM columns between regions
    const uint32_t raw0 = smem_addr(smem_raw);
    const uint32_t base = (raw0 + 1023u) & ~1023u;
    const uint32_t QBOXB = (uint32_t)NQ * 128;  // one half (64 columns) of all NQ query rows
    const uint32_t Qs = base;
    const uint32_t Ks = base + HALVES * QBOXB;
    // per epilogue warp: the normalisers of its columns, after the K ring
    float *bsh = reinterpret_cast<float *>(smem_raw + (base - raw0) + HALVES * QBOXB + (size_t)NS * KSTAGE);
    auto init_barriers = [&](int first, int step) {
        if (first == 0) {
            prefetch_tensormap(&tmQ);
            prefetch_tensormap(&tmK);
            mbar_init(smem_addr(&bar_qfull), 1);
            mbar_init(smem_addr(&bar_qempty), 1);
            abort_sh = 0;
        }
        for (int s = first; s < NS; s += step) {
            mbar_init(smem_addr(&bar_kfull[s]), 1);
            mbar_init(smem_addr(&bar_kempty[s]), 1);
        }
        for (int b = first; b < NR; b += step) {
            mbar_init(smem_addr(&bar_afull[b]), 1);
            mbar_init(smem_addr(&bar_aempty[b]), 4 * split);
        }
        for (int k = first; k < 4 * sets * kP2Slots; k += step)
            mbar_init(smem_addr(&bar_part[k / kP2Slots][k % kP2Slots]), split - 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_shared();
    };
    if constexpr (SHORT) {
        if (warp == 0) init_barriers(lane, 32);
    } else {
        if (tid == 0) init_barriers(0, 1);
    }
    if (warp == 1) {
        tmem_alloc(smem_addr(&tmem_sh), kTmemCols);
        tmem_relinquish();
    }
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_sh;
    volatile int *abort_flag = &abort_sh;
    // everything above runs while the previous kernel drains; from here on its outputs
    // (lens, the row normalisers, the window queries) are read
    wait_prior_grid();

    bool ok = true;
    int s = 0, kph = 0, nq = 0, gt = 0;  // K stage and its parity; query loads; tiles
    int b = 0, aph = 0, done = 0;        // accumulator region and its parity; tiles summed by this warp
    auto next_region = [&](int n) {
        for (; n > 0; --n)
            if (++b == NR) {
                b = 0;
                aph ^= 1;
            }
    };
    for (int skip = 0, n_runs = 1; skip < n_runs; skip += kPlanRuns) {
        // with the normalisers given, this is the call's only pass: it reports lengths out of range
        unsigned *err_len = row_lse != nullptr ? err : nullptr;
        if constexpr (SHORT)
            n_runs = plan_runs<4>(plan, lens, mask, w, L_cap, units, true, kTile, skip, ulist, ucount, err_len);
        else
            n_runs = plan_runs_call(plan, lens, mask, w, L_cap, units, true, kTile, skip, ulist, ucount, err_len);
        const int n_here = min(kPlanRuns, n_runs - skip);
        if (warp == 0) {  // producer
            const int qbox_rows = NQ > 256 ? NQ / 2 : NQ;
            for (int e = 0; ok && e < n_here; ++e) {
                const TileRun run = plan.run[e];
                if (nq > 0 && !(ok = warp_wait(smem_addr(&bar_qempty), (nq - 1) & 1, abort_flag, err))) break;
                if (elect_one()) {
                    const long lb = run.u / Hkv;
                    const int q_row0 = (int)((lb * Hq + (run.u % Hkv) * G) * w);
                    mbar_expect_tx(smem_addr(&bar_qfull), HALVES * QBOXB);
                    for (int hh = 0; hh < HALVES; ++hh)
                        for (int r0 = 0; r0 < NQ; r0 += qbox_rows)
                            tma_load_2d(Qs + hh * QBOXB + r0 * 128, &tmQ, 64 * hh, q_row0 + r0, smem_addr(&bar_qfull));
                }
                ++nq;
                const int k_row0 = run.u * L_cap + run.t0 * kTile;
                for (int t = 0; t < run.nt; ++t) {
                    if (!(ok = warp_wait(smem_addr(&bar_kempty[s]), kph ^ 1, abort_flag, err))) break;
                    if (elect_one()) {
                        mbar_expect_tx(smem_addr(&bar_kfull[s]), KSTAGE);
                        for (int hh = 0; hh < HALVES; ++hh)
                            tma_load_2d(Ks + s * KSTAGE + hh * KBOX, &tmK, 64 * hh, k_row0 + t * kTile,
                                        smem_addr(&bar_kfull[s]));
                    }
                    if (++s == NS) {
                        s = 0;
                        kph ^= 1;
                    }
                }
            }
        } else if (warp == 1) {  // MMA issuer: one chain per piece
            const uint32_t idesc = idesc_bf16(128, NW);
            const uint64_t bh16 = (uint64_t)(QBOXB >> 4);
            for (int e = 0; ok && e < n_here; ++e) {
                const int nt = plan.run[e].nt;
                if (!(ok = warp_wait(smem_addr(&bar_qfull), nq & 1, abort_flag, err))) break;
                ++nq;
                for (int t = 0; ok && t < nt; ++t) {
                    if (!(ok = warp_wait(smem_addr(&bar_kfull[s]), kph, abort_flag, err))) break;
                    for (int h = 0; h < NP; ++h) {
                        if (!(ok = warp_wait(smem_addr(&bar_aempty[b]), aph ^ 1, abort_flag, err))) break;
                        tc_fence_after();
                        // descriptors of the first K slice; later slices add their offset / 16
                        const uint32_t d = tmem + (uint32_t)(b * stride);
                        const uint64_t ad0 = sw128_desc(Ks + s * KSTAGE);
                        const uint64_t bd0 = sw128_desc(Qs + h * NW * 128);
                        auto issue = [&](int k) {
                            const int hh = k >> 2, kk = k & 3;
                            tc_mma(d, ad0 + (uint64_t)((hh * KBOX + kk * 32) >> 4),
                                   bd0 + hh * bh16 + (uint64_t)(kk * 2), idesc, k > 0 ? 1u : 0u);
                        };
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < D / 16; ++k) issue(k);
                            tc_commit(smem_addr(&bar_afull[b]));
                            if (h == NP - 1) {
                                tc_commit(smem_addr(&bar_kempty[s]));
                                if (t == nt - 1) tc_commit(smem_addr(&bar_qempty));
                            }
                        }
                        __syncwarp();
                        next_region(1);
                    }
                    if (++s == NS) {
                        s = 0;
                        kph ^= 1;
                    }
                }
            }
        } else {  // epilogue: set g sums every sets-th key tile, one key per thread
            const int g = ((warp - 2) >> 2) / split, range = ((warp - 2) >> 2) % split, quarter = warp & 3;
            const float invG = 1.f / (float)G;
            const int c_lo = split8_lo(NW, split, range), nc = split8_lo(NW, split, range + 1) - c_lo;  // its columns
            float *bs = bsh + ((g * NP * NW + NP * c_lo) * 4 + quarter * NP * nc);
            for (int e = 0; ok && e < n_here; ++e) {
                const TileRun run = plan.run[e];
                int t = (g - gt) & (sets - 1), cur = 0;  // this set's next tile; the tile region b belongs to
                if (t < run.nt) {  // this unit's row normalisers (warp-private copy); +inf for padding
                    __syncwarp();  // columns, which then add exp2(-inf) = 0
                    for (int h = 0; h < NP; ++h)
                        for (int c = lane; c < nc; c += 32) {
                            const int rr = h * NW + c_lo + c;
                            float bv = INFINITY;
                            if (rr < R) {
                                if (row_lse != nullptr) {  // row (g, t) of the window: the decode's lse of that query
                                    const long qi = (long)(run.u / Hkv) * Hq + (run.u % Hkv) * G + rr / w;
                                    const float l = row_lse[(long)(rr % w) * rows_q + qi];
                                    if (isfinite(l)) {
                                        bv = l * kLog2e;
                                    } else {  // the row adds nothing; the device error word says why
                                        raise_error(err, ERR_NORM);
                                    }
                                } else {
                                    bv = rowb[(long)run.u * R + rr];
                                }
                            }
                            bs[h * nc + c] = bv;
                        }
                    __syncwarp();
                }
                for (; t < run.nt; t += sets) {
                    next_region((t - cur) * NP);
                    cur = t + 1;
                    float a4[4] = {0.f, 0.f, 0.f, 0.f};
                    for (int h = 0; h < NP; ++h) {
                        if (!(ok = warp_wait(smem_addr(&bar_afull[b]), aph, abort_flag, err))) break;
                        tc_fence_after();
                        uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * stride + c_lo);
                        const float *bh = bs + h * nc;
                        auto release = [&]() {  // after this warp's last load of the region
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(smem_addr(&bar_aempty[b]));
                        };
                        float v0[16], v1[16];
                        int left = nc;
                        if (left >= 16) {
                            tmem_ld16_nowait(ta, v0);
                            while (colsum_step(ta, bh, left, v0, v1, c2, a4, release) &&
                                   colsum_step(ta, bh, left, v1, v0, c2, a4, release)) {
                            }
                        } else {  // 8 columns
                            tmem_ld8_nowait(ta, v0);
                            colsum_norms<8>(bh, v1);
                            tmem_ld_wait_regs<8>(v0);
                            release();
                            colsum_batch<8>(v0, v1, c2, a4);
                        }
                        next_region(1);
                    }
                    if (!ok) break;
                    float sum = (a4[0] + a4[1]) + (a4[2] + a4[3]);
                    // the other ranges' sums reach the first range's warp through a slot: it cannot be
                    // refilled before it is read, since a region's release needs every range's warps
                    const int sl = done % kP2Slots, par = (done / kP2Slots) & 1;
                    float(*slot)[32] = &part_sh[((g * 4 + quarter) * kP2Slots + sl) * (split - 1)];
                    const uint32_t bar = smem_addr(&bar_part[g * 4 + quarter][sl]);
                    ++done;
                    if (range) {
                        slot[range - 1][lane] = sum;
                        __syncwarp();
                        if (lane == 0) mbar_arrive(bar);
                        continue;
                    }
                    if (!(ok = warp_wait(bar, par, abort_flag, err))) break;
                    for (int k = 0; k + 1 < split; ++k) sum += slot[k][lane];
                    const int j = (run.t0 + t) * kTile + quarter * 32 + lane;
                    if (j < run.L - w) raw[(long)run.u * L_cap + j] = sum * invG;
                }
                next_region((run.nt - cur) * NP);
                gt += run.nt;
            }
        }
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

// ---------------------------------------------------------------- host side

// Pass 2's pieces: NQ = R rounded up to 16 (to 32 above 256 rows), one MMA chain of N = NQ
// per key tile, or two of N = NQ / 2 above 256 rows; NR TMEM regions of those columns.
struct P2Shape {
    int NQ, NP, NR;
};
static P2Shape p2_shape(int R)
{
    P2Shape p;
    p.NQ = R > 256 ? ((R + 31) / 32) * 32 : ((R + 15) / 16) * 16;
    p.NP = p.NQ > 256 ? 2 : 1;
    const int nw = p.NQ / p.NP;
    p.NR = min(4, kTmemCols / p2_stride(nw));
    return p;
}

bool score_tc_supported(const reco_kv &kv, int w)
{
    const long long R = (long long)(kv.H_q / kv.H_kv) * w;
    const unsigned long long k_rows = (unsigned long long)kv.n_layers * kv.B * kv.H_kv * kv.L_cap;
    const unsigned long long q_rows = (unsigned long long)kv.n_layers * kv.B * kv.H_q * w;
    return kv.dtype == RECO_BF16 && (kv.d == 64 || kv.d == 128) && R <= kTcMaxR && k_rows < (1ull << 31) &&
           q_rows < (1ull << 31);
}

// Pass-1 partials per chunk for R window rows (the combine merges them): the EG of pass1_by_mt.
int score_tc_pass1_groups(int R) { return (R + 127) / 128 <= 2 ? 2 : 1; }

template <int D, int MT, int EG, bool SPLIT = false>
static cudaError_t run_pass1(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask, int w,
                             float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool *ok)
{
    using C = Pass1Cfg<D, MT, EG, SPLIT>;
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const int R = (kv.H_q / kv.H_kv) * w;
    const int nch = (kv.L_cap + kScoreChunk - 1) / kScoreChunk;
    const unsigned long long k_rows = (unsigned long long)units * kv.L_cap;
    const unsigned long long q_rows = (unsigned long long)kv.n_layers * kv.B * kv.H_q * w;
    CUtensorMap mq, mk;
    if (!encode_bf16_2d(&mq, q_win, q_rows, D, 64, 128) || !encode_bf16_2d(&mk, kv.k, k_rows, D, 64, kTile)) {
        *ok = false;
        return cudaSuccess;
    }
    cudaError_t e = allow_smem((const void *)score_rowstats_tc<D, MT, EG, SPLIT>, (int)C::SMEM);
    if (e != cudaSuccess) return e;
    const int grid = (int)min(plan_items(units, kv.L_cap, kScoreChunk), (long long)device_sm_count());
    e = launch_pdl(score_rowstats_tc<D, MT, EG, SPLIT>, dim3(grid), dim3(C::THREADS), C::SMEM, s, mq, mk, lens, mask, w,
                   kv.H_q / kv.H_kv, kv.H_q, kv.H_kv, kv.L_cap, R, nch, (int)units, c2, ws.part_m, ws.part_z, err);
    *ok = true;
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int D>
static cudaError_t pass1_by_mt(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask, int w,
                               float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool *ok)
{
    const int MT = ((kv.H_q / kv.H_kv) * w + 127) / 128;
    if (kv.L_cap <= kSplitCap && MT <= 2)
        return MT == 1 ? run_pass1<D, 1, 2, true>(kv, q_win, lens, mask, w, c2, ws, err, s, ok)
                       : run_pass1<D, 2, 2, true>(kv, q_win, lens, mask, w, c2, ws, err, s, ok);
    switch (MT) {
    case 1: return run_pass1<D, 1, 2>(kv, q_win, lens, mask, w, c2, ws, err, s, ok);
    case 2: return run_pass1<D, 2, 2>(kv, q_win, lens, mask, w, c2, ws, err, s, ok);
    case 3: return run_pass1<D, 3, 1>(kv, q_win, lens, mask, w, c2, ws, err, s, ok);
    default: return run_pass1<D, 4, 1>(kv, q_win, lens, mask, w, c2, ws, err, s, ok);
    }
}

cudaError_t launch_score_tc_pass1(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask,
                                  int w, float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool *used)
{
    *used = false;
    if (!score_tc_supported(kv, w)) return cudaSuccess;
    return kv.d == 128 ? pass1_by_mt<128>(kv, q_win, lens, mask, w, c2, ws, err, s, used)
                       : pass1_by_mt<64>(kv, q_win, lens, mask, w, c2, ws, err, s, used);
}

template <int D>
static cudaError_t run_pass2(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask, int w,
                             float c2, const ScoreWs &ws, const float *row_lse, unsigned *err, cudaStream_t s,
                             bool *ok)
{
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const int R = (kv.H_q / kv.H_kv) * w;
    const P2Shape ps = p2_shape(R);
    const unsigned long long k_rows = (unsigned long long)units * kv.L_cap;
    const unsigned long long q_rows = (unsigned long long)kv.n_layers * kv.B * kv.H_q * w;
    CUtensorMap mq, mk;
    const int qbox = ps.NQ > 256 ? ps.NQ / 2 : ps.NQ;
    if (!encode_bf16_2d(&mq, q_win, q_rows, D, 64, qbox) || !encode_bf16_2d(&mk, kv.k, k_rows, D, 64, kTile)) {
        *ok = false;
        return cudaSuccess;
    }
    const long long tiles = plan_items(units, kv.L_cap, kTile);
    const int grid = (int)min(tiles, (long long)device_sm_count());
    // two sets where they stay apart (a set's pieces of consecutive turns lie NP + 1 apart), and where a tile's
    // columns are too few for all groups
    const int sets = ps.NQ / ps.NP < 8 * kP2Groups || (ps.NP + 1 <= ps.NR && tiles > grid) ? 2 : 1;
    const size_t qbytes = (size_t)(D / 64) * ps.NQ * 128, kstage = (size_t)(D / 64) * kTile * 128;
    const size_t nbytes = (size_t)4 * sets * ps.NQ * sizeof(float);  // the epilogue warps' normalisers
    const size_t budget = 227 * 1024 - (sizeof(TilePlan) + 7 * 1024) - 1024;
    if (qbytes + nbytes + 2 * kstage > budget) {
        *ok = false;
        return cudaSuccess;
    }
    const int NS = (int)min((size_t)4, (budget - qbytes - nbytes) / kstage);
    const size_t smem = 1024 + qbytes + (size_t)NS * kstage + nbytes;
    auto colsum = tiles <= (long long)kShortTiles * grid ? score_colsum_tc<D, true> : score_colsum_tc<D, false>;
    cudaError_t e = allow_smem((const void *)colsum, (int)smem);
    if (e != cudaSuccess) return e;
    const bool masked = mask.keep != nullptr;
    e = launch_pdl(colsum, dim3(grid), dim3(64 + 128 * kP2Groups), smem, s, mq, mk, lens, mask, w,
                   kv.H_q / kv.H_kv, kv.H_q, kv.H_kv, kv.L_cap, R, ps.NQ, ps.NP, ps.NR, NS, sets, (int)units, c2,
                   (const float *)ws.rowb, row_lse, (long)kv.n_layers * kv.B * kv.H_q, ws.raw,
                   masked ? ws.ulist : nullptr, masked ? ws.ucount : nullptr, err);
    *ok = true;
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_score_tc_pass2(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask,
                                  int w, float c2, const ScoreWs &ws, const float *row_lse, unsigned *err,
                                  cudaStream_t s, bool *used)
{
    *used = false;
    if (!score_tc_supported(kv, w)) return cudaSuccess;
    return kv.d == 128 ? run_pass2<128>(kv, q_win, lens, mask, w, c2, ws, row_lse, err, s, used)
                       : run_pass2<64>(kv, q_win, lens, mask, w, c2, ws, row_lse, err, s, used);
}

}  // namespace reco
