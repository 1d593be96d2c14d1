// decode.cu -- decode attention over the ragged compacted cache, the per-token
// attention whose cost the compression lowers (Sec. 1; Sec. 2.2; Sec. 4.2).
//
// decode_stream: a persistent split-K flash-decode, one CTA of 8 warps per SM (for long
// bf16 work 4 of them, each with a ring twice as deep).  Every CTA first builds the same
// work plan from lens: the prefix sum of blocks of keys per unit, with the blocks of all
// units laid end to end and cut into one equal contiguous range per warp (a stream-K
// split: balanced to one block, no work queue).  A call with more units than one plan
// holds runs as consecutive launches over contiguous unit ranges.  When no unit is long
// enough to be cut, the units are instead sorted by length and dealt whole to the warps in
// snake order (longest first).  An item's keys stream from HBM in blocks of 8 KB (at d =
// 128): one lane issues bulk copies of K and V into the warp's 3-stage ring and the warp
// waits on the stage's mbarrier (bounded).  What a warp does with a block is a template
// parameter, a block consumer.
//   bf16: blocks of 16 keys by TMA tensor copies (128-byte swizzled 16 x 64 tiles); QK^T
//   and PV on mma.sync m16n8k16 (fp32 accumulate), up to 16 query heads.  The head
//   dimension is permuted consistently on the Q and K sides (and on the V and output
//   sides) so that each thread's fragments are whole 16-byte chunks, and the swizzle makes
//   every fragment read conflict-free.  A unit of 9 to 16 heads runs as two units of half the
//   heads (28 x 4 x 4 units of 2000 to 4100 rows, 16 heads: 215 -> 128 us from half the warps
//   with deep rings to all of them); with many short units its other heads fill the QK tile's
//   other eight rows instead, one pass over the block.
//   float32: blocks of 8 keys, plain FMAs (28 x 4 x 2 units of 800 to 1500 rows, 6 heads,
//   from one CTA per unit that took its keys one by one: 540 -> 61 us).
// A unit split over several items writes partial (max, sum, output) triples; the last
// item to finish (atomic ticket, no waiting) merges them.  The counters live in the
// caller's workspace, zero-filled before its first use; each launch clears what it
// counted, so no reset runs between launches.  The appended token (k_new, v_new) is
// read from the inputs and written into the cache by the warp that covers its index;
// the last warp of the grid to finish advances lens.
//
// decode_simt serves bf16 calls for which no tensor map can be made.
#include <cuda.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "internal.h"
#include "tma.cuh"

namespace reco {

DecodeWs decode_ws_layout(const reco_kv &kv, void *base)
{
    size_t units = (size_t)kv.n_layers * kv.B * kv.H_kv;
    size_t G = kv.H_q / kv.H_kv;
    char *p = (char *)base;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *r = p ? p + off : nullptr;
        off += align256(bytes);
        return r;
    };
    DecodeWs ws;
    ws.part_slots = kDecodePartSlots;
    // merge tickets per unit; a unit of G > 8 heads may run as two
    ws.counters = (int32_t *)take((2 + units * (G > 8 ? 2 : 1)) * 4);
    ws.part_ml = (float *)take((size_t)ws.part_slots * G * 2 * 4);
    ws.part_o = (float *)take((size_t)ws.part_slots * G * kv.d * 4);
    ws.bytes = off;
    return ws;
}

struct DecodeArgs {
    void *K;
    void *V;
    const void *q;
    const void *k_new;
    const void *v_new;
    int32_t *lens;
    void *out;
    float *lse;
    int32_t *counters;
    float *part_ml;
    float *part_o;
    int units, Hq, Hkv, G, L_cap, append, out_bf16;
    float c2;  // scale * log2(e)
    unsigned *err;
    int hs_min, hs_max;  // virtual units per unit, each of G / hs query heads
    float *ring;      // or nullptr: lse rows ring[*slot] and ring[*slot + slots], each [nq]
    long long *slot;  // device ring row, advanced by one (mod slots) per launch
    int slots;
    long long nq;     // query heads of the launch (layers * B * H_q)
    void *qring;      // or nullptr: [nq][slots][D] of q's dtype, row *slot of every head gets its query
    long long nq_rows;  // query heads of this launch (nq, or a part of it when the units are split)
    int advance;        // this launch advances *slot (the last of a split launch's parts)
};

// The ring row this launch writes (read once the previous kernel's writes are visible),
// or -1 without a ring; a slot outside [0, slots) writes nothing and sets the error word.
__device__ __forceinline__ long long ring_row(const DecodeArgs &a)
{
    if (!a.ring) return -1;
    const long long s = *a.slot;
    if (s < 0 || s >= a.slots) {
        raise_error(a.err, ERR_INTERNAL);
        return -1;
    }
    return s;
}

// lse of query row i: to the lse output and, with a ring, to ring rows rs and rs + slots.
__device__ __forceinline__ void put_lse(const DecodeArgs &a, long long rs, size_t i, float v)
{
    if (a.lse) a.lse[i] = v;
    if (rs >= 0) {
        a.ring[rs * a.nq + (long long)i] = v;
        a.ring[(rs + a.slots) * a.nq + (long long)i] = v;
    }
}

// atomicAdd with acquire-release semantics at GPU scope.
__device__ __forceinline__ int atom_add_acq_rel(int *p, int v)
{
    int old;
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

__device__ __forceinline__ unsigned long long atom_add_acq_rel_u64(unsigned long long *p, unsigned long long v)
{
    unsigned long long old;
    asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
    return old;
}

__device__ __forceinline__ bool unit_ok(int L, int L_cap, int append)
{
    return L >= 0 && L <= L_cap && (!append || L < L_cap);
}

__device__ __forceinline__ void store_out(void *out, bool bf16, size_t i, float v)
{
    if (bf16)
        reinterpret_cast<__nv_bfloat16 *>(out)[i] = __float2bfloat16_rn(v);
    else
        reinterpret_cast<float *>(out)[i] = v;
}

// ---------------------------------------------------------------- SIMT path
template <typename T, int D>
__global__ void __launch_bounds__(128) decode_simt(DecodeArgs a)
{
    constexpr int NW = 4, PER = D / 32, GM = 16;
    __shared__ float sm_m[NW][GM], sm_l[NW][GM];
    __shared__ float sm_o[NW][GM][D];
    const long u = blockIdx.x;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int L = a.lens[u];
    const long long rs = ring_row(a);
    const bool ok = unit_ok(L, a.L_cap, a.append);
    if (!ok && threadIdx.x == 0) raise_error(a.err, (a.append && L == a.L_cap) ? ERR_ROOM : ERR_LEN);
    const int Le = ok ? L + a.append : 0;
    const long lb = u / a.Hkv;
    const int h = (int)(u % a.Hkv);
    const int G = a.G;
    T *Kp = reinterpret_cast<T *>(a.K) + u * (long)a.L_cap * D;
    T *Vp = reinterpret_cast<T *>(a.V) + u * (long)a.L_cap * D;
    const T *kn = a.append ? reinterpret_cast<const T *>(a.k_new) + u * D : nullptr;
    const T *vn = a.append ? reinterpret_cast<const T *>(a.v_new) + u * D : nullptr;
    const T *qp = reinterpret_cast<const T *>(a.q) + (lb * a.Hq + (long)h * G) * D;
    float q[GM][PER], o[GM][PER], m[GM], l[GM];
#pragma unroll
    for (int g = 0; g < GM; ++g) {
        m[g] = -INFINITY;
        l[g] = 0.f;
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            q[g][i] = g < G ? to_float(qp[(long)g * D + lane * PER + i]) : 0.f;
            o[g][i] = 0.f;
        }
    }
    for (int j = wid; j < Le; j += NW) {
        const T *kr = (a.append && j == L) ? kn : Kp + (long)j * D;
        const T *vr = (a.append && j == L) ? vn : Vp + (long)j * D;
        float kk[PER], vv[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            kk[i] = to_float(kr[lane * PER + i]);
            vv[i] = to_float(vr[lane * PER + i]);
        }
#pragma unroll
        for (int g = 0; g < GM; ++g) {
            if (g < G) {
                float s = 0.f;
#pragma unroll
                for (int i = 0; i < PER; ++i) s = fmaf(q[g][i], kk[i], s);
                s = warp_sum(s) * a.c2;
                const float mn = fmaxf(m[g], s);
                const float al = fast_exp2(m[g] - mn);
                const float p = fast_exp2(s - mn);
                l[g] = l[g] * al + p;
#pragma unroll
                for (int i = 0; i < PER; ++i) o[g][i] = fmaf(o[g][i], al, p * vv[i]);
                m[g] = mn;
            }
        }
    }
#pragma unroll
    for (int g = 0; g < GM; ++g) {
        if (g < G) {
            if (lane == 0) {
                sm_m[wid][g] = m[g];
                sm_l[wid][g] = l[g];
            }
#pragma unroll
            for (int i = 0; i < PER; ++i) sm_o[wid][g][lane * PER + i] = o[g][i];
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < G * D; e += blockDim.x) {
        const int g = e / D, dd = e % D;
        float M = -INFINITY;
        for (int w = 0; w < NW; ++w) M = fmaxf(M, sm_m[w][g]);
        float Ls = 0.f, O = 0.f;
        if (M != -INFINITY) {
            for (int w = 0; w < NW; ++w) {
                const float wt = fast_exp2(sm_m[w][g] - M);
                Ls += sm_l[w][g] * wt;
                O += sm_o[w][g][dd] * wt;
            }
        }
        const size_t row = (size_t)(lb * a.Hq + (long)h * G + g);
        store_out(a.out, a.out_bf16, row * D + dd, Ls > 0.f ? O / Ls : 0.f);
        if (dd == 0) put_lse(a, rs, row, Ls > 0.f ? (M + log2f(Ls)) * kLn2 : -INFINITY);
    }
    if (ok && a.append) {
        for (int e = threadIdx.x; e < D; e += blockDim.x) {
            Kp[(long)L * D + e] = kn[e];
            Vp[(long)L * D + e] = vn[e];
        }
        if (threadIdx.x == 0) a.lens[u] = L + 1;
    }
}

// ---------------------------------------------------------------- streamed path
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// (a, b) -> bf16x2 hi = round(a, b) and lo = round((a, b) - hi).
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t &hi, uint32_t &lo)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    const float2 f = __bfloat1622float2(h);
    hi = *reinterpret_cast<uint32_t *>(&h);
    lo = pack_bf16(a - f.x, b - f.y);
}

__device__ __forceinline__ uint32_t word(const uint4 &v, int x)
{
    return x == 0 ? v.x : (x == 1 ? v.y : (x == 2 ? v.z : v.w));
}

constexpr int kDecodeWarps = 8;       // warps per CTA (one CTA per SM)
constexpr int kDecodeStages = 3;      // ring stages per warp
constexpr int kMaxTmaUnits = 8192;    // one plan entry per unit kept in shared memory
constexpr long long kSpinLimit = 1LL << 24;  // bounded mbarrier waits (about a second)
constexpr float kLazyLog2 = 8.f;             // output rescale threshold (log2 units)
constexpr int kMinBlocksPerWarp = 4;         // fewer working warps rather than shorter ranges
constexpr int kCheapPieces = 8;              // pieces of a unit that are merged without a thought
constexpr int kMaxWholeBlocks = 16;          // units of at most this many blocks are never cut
constexpr int kOnePassBlocks = 16;           // blocks per warp from which all heads of a unit may run in one pass
// units from which they may, of `warps` warps
__host__ __device__ constexpr int one_pass_units(int warps) { return warps * 2 / 3; }
constexpr int kDeepBlocksPerWarp = 64;       // from this many blocks per warp, half the warps with deep rings

constexpr int kStageBytes128 = 8192;         // a block of K and V rows at d = 128 (half of it at d = 64)

template <int D> struct RingLayout {
    static constexpr int STAGE = kStageBytes128 * D / 128;
    static constexpr int RING = kDecodeWarps * kDecodeStages * STAGE;
};

// the largest plan fits beside the d = 128 ring (227 KB per CTA, about 1 KB of it static, for
// float32 about 3 KB)
constexpr int kMaxF32Units = kMaxTmaUnits - 1024;
static_assert(1024 + RingLayout<128>::RING + (kMaxTmaUnits + 1) * 4 + 1024 <= 227 * 1024, "decode smem budget");
static_assert(1024 + RingLayout<128>::RING + (kMaxF32Units + 1) * 4 + 4 * 1024 <= 227 * 1024, "decode smem budget");
static_assert((kMaxTmaUnits + 32 + (kMaxWholeBlocks + 1) * kDecodeWarps * 32) * 4 <= RingLayout<64>::RING,
              "lengths and the sort counters are staged in the ring");

template <int D>
size_t ring_smem_bytes(int units)
{
    return 1024 + (size_t)RingLayout<D>::RING + (size_t)(units + 1) * sizeof(int);
}

// Byte offset of 16-byte chunk ch (0..7) of row rr inside a 128B-swizzled 16-row box.
__device__ __forceinline__ uint32_t swz(int rr, int ch) { return rr * 128 + ((ch ^ (rr & 7)) << 4); }

// A block consumer holds one item's queries, running (max, sum) and output in a warp's registers
// and takes the item's keys in blocks of KB rows from the warp's ring.  It says how a block is
// copied (load), where a 16-byte chunk of a row lies in a stage (chunk), and how results leave.

// bf16: QK^T and PV run on mma.sync m16n8k16 with NT * 8 query heads per unit.  The QK tile has
// 16 query rows: heads 0-7 fill its first eight, heads 8-15 (NT = 2) the others, which cost the
// product nothing more; PV takes one 8-head column tile per NT.
template <class T> struct Tag {
    using type = T;
};

template <int D_, int NT_, int HALVES_ = 1> struct Bf16Block {
    static constexpr int D = D_, NT = NT_, KB = 16, GM = 8 * NT;
    // units run as two halves of their heads (HALVES = 2), or may (NT = 2): then by consumer Half
    static constexpr bool SPLIT = NT == 2 || HALVES_ == 2, ALWAYS = HALVES_ == 2;
    using Half = Bf16Block<D_, 1, HALVES_>;
    static constexpr int ROW = 2 * D, HALVES = D / 64, TILE = 16 * 128, MT = D / 16;
    static constexpr int APP = (2 * ROW / 16 + 31) / 32, SCRATCH = 0;
    static constexpr bool TENSOR_MAPS = true, PREFETCH_Q = NT == 1;
    // half the warps with deeper rings for long work: with up to eight heads a block leaves a warp
    // waiting for data
    static constexpr bool DEEP = true;

    uint32_t qa[D / 16][2 * NT], qn[PREFETCH_Q ? D / 16 : 1][2 * NT];
    float o[NT][MT][4], m[NT], l[NT];
    const __nv_bfloat16 *q_src = nullptr;
    int nh_src = 0;
    const int g, c;

    static_assert(NT_ == 1 || HALVES_ == 1, "sixteen heads need no halves");
    __device__ __forceinline__ Bf16Block(int lane, float *) : g(lane >> 2), c(lane & 3) {}

    __device__ static __forceinline__ uint32_t chunk(int row, int ch) { return (ch >> 3) * TILE + swz(row, ch & 7); }

    // 128-byte swizzled 16 x 64 boxes of K, then of V (whole boxes: rows past the item are masked)
    __device__ static __forceinline__ void load(uint32_t dst, uint32_t bar, const CUtensorMap *tmK,
                                                const CUtensorMap *tmV, const DecodeArgs &a, int pu, int k, int,
                                                uint64_t policy)
    {
        const int y = pu * a.L_cap + k;
        mbar_expect_tx(bar, 2 * HALVES * TILE);
#pragma unroll
        for (int hh = 0; hh < HALVES; ++hh) {
            tma_load_2d_hint(dst + hh * TILE, tmK, 64 * hh, y, bar, policy);
            tma_load_2d_hint(dst + (HALVES + hh) * TILE, tmV, 64 * hh, y, bar, policy);
        }
    }

    // Q fragments, the head dim permuted to match the K chunks: k-step j = 4*hh + 2*e + half takes
    // elements 64*hh + 16c + 8e + 4*half + {0,1} and + {2,3} (of rows g, then g + 8)
    __device__ __forceinline__ void fragments(const __nv_bfloat16 *q, int nh, uint32_t (&f)[D / 16][2 * NT]) const
    {
#pragma unroll
        for (int hh = 0; hh < HALVES; ++hh)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    uint4 wv = make_uint4(0, 0, 0, 0);
                    if (g + 8 * n < nh) wv = *reinterpret_cast<const uint4 *>(q + (g + 8 * n) * D + 64 * hh + 16 * c + 8 * e);
                    const int j = 4 * hh + 2 * e;
                    f[j][n] = wv.x;
                    f[j][NT + n] = wv.y;
                    f[j + 1][n] = wv.z;
                    f[j + 1][NT + n] = wv.w;
                }
    }

    // the queries of the item that start() will begin
    __device__ __forceinline__ void load_q(const void *q, long qrow, int nh)
    {
        q_src = reinterpret_cast<const __nv_bfloat16 *>(q) + qrow * D;
        nh_src = nh;
        if constexpr (PREFETCH_Q) fragments(q_src, nh, qn);
    }

    __device__ __forceinline__ void start()
    {
        if constexpr (PREFETCH_Q) {
#pragma unroll
            for (int j = 0; j < D / 16; ++j)
#pragma unroll
                for (int n = 0; n < 2 * NT; ++n) qa[j][n] = qn[j][n];
        } else {
            fragments(q_src, nh_src, qa);
        }
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            m[n] = -INFINITY;
            l[n] = 0.f;
#pragma unroll
            for (int t = 0; t < MT; ++t) o[n][t][0] = o[n][t][1] = o[n][t][2] = o[n][t][3] = 0.f;
        }
    }

    __device__ __forceinline__ void consume(uint32_t Ks, uint32_t Vs, int kb, int k1, float c2)
    {
        // four accumulators (keys 0-7 / 8-15, even / odd k-steps): dependent MMA chains
        // of D/32 instead of D/16
        float s0[4] = {0.f, 0.f, 0.f, 0.f}, s1[4] = {0.f, 0.f, 0.f, 0.f};
        float t0[4] = {0.f, 0.f, 0.f, 0.f}, t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int hh = 0; hh < HALVES; ++hh)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const uint4 ka = lds_u4(Ks + hh * TILE + swz(g, 2 * c + e));
                const uint4 kc = lds_u4(Ks + hh * TILE + swz(8 + g, 2 * c + e));
                const int j = 4 * hh + 2 * e;
                const uint32_t a1 = NT == 2 ? qa[j][1 % (2 * NT)] : 0u, a3 = NT == 2 ? qa[j][3 % (2 * NT)] : 0u;
                const uint32_t b1 = NT == 2 ? qa[j + 1][1 % (2 * NT)] : 0u, b3 = NT == 2 ? qa[j + 1][3 % (2 * NT)] : 0u;
                mma_bf16(s0, qa[j][0], a1, qa[j][NT], a3, ka.x, ka.y);
                mma_bf16(s1, qa[j][0], a1, qa[j][NT], a3, kc.x, kc.y);
                mma_bf16(t0, qa[j + 1][0], b1, qa[j + 1][NT], b3, ka.z, ka.w);
                mma_bf16(t1, qa[j + 1][0], b1, qa[j + 1][NT], b3, kc.z, kc.w);
            }
        uint32_t ph[NT][2], pl[NT][2];
        const int kA = kb + 2 * c, kB = kb + 8 + 2 * c;
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            // scores of query g + 8n for keys kb+2c, kb+2c+1, kb+8+2c, kb+9+2c
            const float x0 = (kA < k1) ? (s0[2 * n] + t0[2 * n]) * c2 : -INFINITY;
            const float x1 = (kA + 1 < k1) ? (s0[2 * n + 1] + t0[2 * n + 1]) * c2 : -INFINITY;
            const float x2 = (kB < k1) ? (s1[2 * n] + t1[2 * n]) * c2 : -INFINITY;
            const float x3 = (kB + 1 < k1) ? (s1[2 * n + 1] + t1[2 * n + 1]) * c2 : -INFINITY;
            float mb = fmaxf(fmaxf(x0, x1), fmaxf(x2, x3));
            mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, 1));
            mb = fmaxf(mb, __shfl_xor_sync(0xffffffffu, mb, 2));
            // Lazy rescale: a row's reference max m moves only when a block max exceeds it
            // by more than 2^kLazyLog2, so probabilities against a stale m stay <= 2^8
            // (exact in fp32, and the bf16 hi + lo split keeps 16 bits of them); the
            // output rescale below then runs on few blocks.  m, l and o stay consistent, so
            // o / l and lse = m + log2 l are the same quantities as with an exact max.
            const bool grow = mb > m[n] + kLazyLog2;
            if (__any_sync(0xffffffffu, grow)) {
                const float mn = grow ? mb : m[n];
                const float alpha = grow ? fast_exp2(m[n] - mn) : 1.f;  // m = -inf gives 0
                l[n] *= alpha;
                m[n] = mn;
                const float al0 = __shfl_sync(0xffffffffu, alpha, (2 * c) * 4);
                const float al1 = __shfl_sync(0xffffffffu, alpha, (2 * c + 1) * 4);
#pragma unroll
                for (int t = 0; t < MT; ++t) {
                    o[n][t][0] *= al0;
                    o[n][t][1] *= al1;
                    o[n][t][2] *= al0;
                    o[n][t][3] *= al1;
                }
            }
            const float base = (m[n] == -INFINITY) ? 0.f : m[n];
            const float p0 = fast_exp2(x0 - base), p1 = fast_exp2(x1 - base);
            const float p2 = fast_exp2(x2 - base), p3 = fast_exp2(x3 - base);
            l[n] += (p0 + p1) + (p2 + p3);
            // P enters the PV product as bf16 hi + lo parts (two MMAs), which keeps about
            // 16 significant bits of each probability instead of 8.
            split_bf16(p0, p1, ph[n][0], pl[n][0]);
            split_bf16(p2, p3, ph[n][1], pl[n][1]);
        }
#pragma unroll
        for (int hh = 0; hh < HALVES; ++hh) {
            const uint4 v0 = lds_u4(Vs + hh * TILE + swz(2 * c, g));
            const uint4 v1 = lds_u4(Vs + hh * TILE + swz(2 * c + 1, g));
            const uint4 v2 = lds_u4(Vs + hh * TILE + swz(2 * c + 8, g));
            const uint4 v3 = lds_u4(Vs + hh * TILE + swz(2 * c + 9, g));
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                const uint32_t W0 = word(v0, x), W1 = word(v1, x), W2 = word(v2, x), W3 = word(v3, x);
                const uint32_t A0 = __byte_perm(W0, W1, 0x5410), A1 = __byte_perm(W0, W1, 0x7632);
                const uint32_t A2 = __byte_perm(W2, W3, 0x5410), A3 = __byte_perm(W2, W3, 0x7632);
#pragma unroll
                for (int n = 0; n < NT; ++n) {
                    mma_bf16(o[n][4 * hh + x], A0, A1, A2, A3, ph[n][0], ph[n][1]);
                    mma_bf16(o[n][4 * hh + x], A0, A1, A2, A3, pl[n][0], pl[n][1]);
                }
            }
        }
    }

    __device__ __forceinline__ void finish()
    {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            l[n] += __shfl_xor_sync(0xffffffffu, l[n], 1);
            l[n] += __shfl_xor_sync(0xffffffffu, l[n], 2);
        }
    }

    template <typename F> __device__ __forceinline__ void each_lse(int G, F f) const
    {
#pragma unroll
        for (int n = 0; n < NT; ++n)
            if (c == 0 && g + 8 * n < G) f(g + 8 * n, m[n], l[n]);
    }

    __device__ __forceinline__ void store(void *out, bool bf16, long qrow0, int G) const
    {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int q0 = 8 * n + 2 * c, q1 = q0 + 1;
            const float l0 = __shfl_sync(0xffffffffu, l[n], 8 * c), l1 = __shfl_sync(0xffffffffu, l[n], 8 * c + 4);
            const float inv0 = l0 > 0.f ? 1.f / l0 : 0.f, inv1 = l1 > 0.f ? 1.f / l1 : 0.f;
#pragma unroll
            for (int hh = 0; hh < HALVES; ++hh) {
                const long d0 = 64 * hh + 8 * g;
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    const float *v = o[n][4 * hh + x];
                    if (q0 < G) {
                        store_out(out, bf16, (qrow0 + q0) * D + d0 + 2 * x, v[0] * inv0);
                        store_out(out, bf16, (qrow0 + q0) * D + d0 + 2 * x + 1, v[2] * inv0);
                    }
                    if (q1 < G) {
                        store_out(out, bf16, (qrow0 + q1) * D + d0 + 2 * x, v[1] * inv1);
                        store_out(out, bf16, (qrow0 + q1) * D + d0 + 2 * x + 1, v[3] * inv1);
                    }
                }
            }
        }
    }

    __device__ __forceinline__ void store_partial(float *po, int G) const
    {
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int q0 = 8 * n + 2 * c, q1 = q0 + 1;
#pragma unroll
            for (int hh = 0; hh < HALVES; ++hh) {
                const int d0 = 64 * hh + 8 * g;
                const float(*v)[4] = &o[n][4 * hh];
                if (q0 < G) {
                    float4 *dst = reinterpret_cast<float4 *>(po + (size_t)q0 * D + d0);
                    dst[0] = make_float4(v[0][0], v[0][2], v[1][0], v[1][2]);
                    dst[1] = make_float4(v[2][0], v[2][2], v[3][0], v[3][2]);
                }
                if (q1 < G) {
                    float4 *dst = reinterpret_cast<float4 *>(po + (size_t)q1 * D + d0);
                    dst[0] = make_float4(v[0][1], v[0][3], v[1][1], v[1][3]);
                    dst[1] = make_float4(v[2][1], v[2][3], v[3][1], v[3][3]);
                }
            }
        }
    }
};

// float32: plain FMAs in float32 throughout, GT >= G (or half of G) query heads.  In QK^T
// lane (kq = lane / 8, part = lane % 8) holds D / 8 elements of every head's query (32-element
// groups, four at part * 4) and multiplies them with keys kq and kq + 4 of the block; the eight
// parts are then added by halving exchanges that leave each (key, head) sum in one lane.  In PV a
// lane owns D / 32 columns of every head's output and takes the probabilities from shared memory.
template <int D_, int GT_> struct F32Block {
    static constexpr int D = D_, KB = 8, GM = GT_, GT = GT_, E = D / 32, QE = D / 8;
    static constexpr int ROW = 4 * D;
    static constexpr bool SPLIT = GT == 8, ALWAYS = false;  // units of more than 8 heads run as two halves
    using Half = F32Block;
    static constexpr int APP = (2 * ROW / 16 + 31) / 32, SCRATCH = KB * GT;
    static constexpr bool TENSOR_MAPS = false;
    static constexpr bool DEEP = false;  // bound by its arithmetic: all the warps (93 against 70 us)
    static constexpr int GP = GT == 8 ? 4 : GT;  // heads per turn of the PV product
    static constexpr int VPL = GT == 8 ? 2 : (GT == 6 ? 3 : 1);  // (key, head) sums per lane

    float q[GT][QE], o[GT][E], m[VPL], l[VPL];
    const float *q_src = nullptr;
    int nh_src = 0;
    float *const p_sm;  // [KB][GT] probabilities of the block
    const int lane;

    __device__ __forceinline__ F32Block(int lane_, float *scratch) : p_sm(scratch), lane(lane_) {}

    __device__ static __forceinline__ uint32_t chunk(int row, int ch) { return row * ROW + ch * 16; }

    // `rows` rows of K, then of V, each one contiguous copy (none when only the appended row is left)
    __device__ static __forceinline__ void load(uint32_t dst, uint32_t bar, const CUtensorMap *, const CUtensorMap *,
                                                const DecodeArgs &a, int pu, int k, int rows, uint64_t policy)
    {
        const uint32_t bytes = (uint32_t)max(rows, 0) * ROW;
        mbar_expect_tx(bar, 2 * bytes);
        if (bytes == 0) return;
        const size_t off = ((size_t)pu * a.L_cap + k) * ROW;
        bulk_load_hint(dst, static_cast<const char *>(a.K) + off, bytes, bar, policy);
        bulk_load_hint(dst + KB * ROW, static_cast<const char *>(a.V) + off, bytes, bar, policy);
    }

    __device__ __forceinline__ void load_q(const void *qp, long qrow, int nh)
    {
        q_src = reinterpret_cast<const float *>(qp) + qrow * D;
        nh_src = nh;
    }

    __device__ __forceinline__ void start()
    {
#pragma unroll
        for (int g = 0; g < GT; ++g) {
#pragma unroll
            for (int i = 0; i < QE / 4; ++i) {
                float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
                if (g < nh_src) x = *reinterpret_cast<const float4 *>(q_src + (long)g * D + 32 * i + 4 * (lane & 7));
                q[g][4 * i] = x.x;
                q[g][4 * i + 1] = x.y;
                q[g][4 * i + 2] = x.z;
                q[g][4 * i + 3] = x.w;
            }
#pragma unroll
            for (int e = 0; e < E; ++e) o[g][e] = 0.f;
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            m[v] = -INFINITY;
            l[v] = 0.f;
        }
    }

    // the lane (of kq = 0, first key) and its value that hold head g after the exchanges
    __device__ static __forceinline__ constexpr int lane_of(int g)
    {
        return GT == 8 ? g >> 1 : (GT == 6 ? 2 * (g / 3) : (GT == 4 ? g : 2 * g));
    }
    __device__ static __forceinline__ constexpr int value_of(int g) { return GT == 8 ? g & 1 : (GT == 6 ? g % 3 : 0); }
    __device__ __forceinline__ int head_of(int v) const
    {
        return GT == 8 ? 2 * (lane & 3) + v : (GT == 4 ? lane & 3 : ((lane >> 1) & 1) * VPL + v);
    }

    // Halving exchange over lane bit `bit`: of 2N partial sums this lane keeps the lower N (bit
    // clear) or the upper N, each with its partner's added.
    template <int N> __device__ __forceinline__ void halve(float *s, int bit) const
    {
        const bool up = lane & bit;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float send = up ? s[i] : s[i + N];
            const float keep = up ? s[i + N] : s[i];
            s[i] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
        }
    }

    __device__ __forceinline__ void consume(uint32_t Ks, uint32_t Vs, int kb, int k1, float c2)
    {
        float s[2 * GT];  // keys kq, then kq + 4
#pragma unroll
        for (int i = 0; i < 2 * GT; ++i) s[i] = 0.f;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const uint32_t row = Ks + ((lane >> 3) + 4 * k) * ROW + (lane & 7) * 16;
#pragma unroll
            for (int i = 0; i < QE / 4; ++i) {
                const float4 x = lds_f4(row + 128 * i);
#pragma unroll
                for (int g = 0; g < GT; ++g) {
                    float t = s[k * GT + g];
                    t = fmaf(q[g][4 * i], x.x, t);
                    t = fmaf(q[g][4 * i + 1], x.y, t);
                    t = fmaf(q[g][4 * i + 2], x.z, t);
                    s[k * GT + g] = fmaf(q[g][4 * i + 3], x.w, t);
                }
            }
        }
        halve<GT>(s, 4);      // lane bit 2: the key
        halve<GT / 2>(s, 2);  // bit 1: the head's high bit
        if constexpr (GT % 4 == 0) {
            halve<GT / 4>(s, 1);
        } else {  // both lanes keep the sums
#pragma unroll
            for (int v = 0; v < VPL; ++v) s[v] += __shfl_xor_sync(0xffffffffu, s[v], 1);
        }
        const int kk = (lane >> 3) + (lane & 4);  // this lane's key of the block
        float x[VPL], mb[VPL];
        bool any = false;
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            x[v] = kb + kk < k1 ? s[v] * c2 : -INFINITY;
            mb[v] = x[v];
#pragma unroll
            for (int o2 = 4; o2 <= 16; o2 <<= 1) mb[v] = fmaxf(mb[v], __shfl_xor_sync(0xffffffffu, mb[v], o2));
            any |= mb[v] > m[v] + kLazyLog2;
        }
        if (__any_sync(0xffffffffu, any)) {  // lazy rescale, as in the bf16 consumer
            float al[VPL];
#pragma unroll
            for (int v = 0; v < VPL; ++v) {
                const float mn = mb[v] > m[v] + kLazyLog2 ? mb[v] : m[v];
                al[v] = mn == m[v] ? 1.f : fast_exp2(m[v] - mn);  // m = -inf gives 0
                l[v] *= al[v];
                m[v] = mn;
            }
#pragma unroll
            for (int g = 0; g < GT; ++g) {
                const float f = __shfl_sync(0xffffffffu, al[value_of(g)], lane_of(g));
#pragma unroll
                for (int e = 0; e < E; ++e) o[g][e] *= f;
            }
        }
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const float p = fast_exp2(x[v] - (m[v] == -INFINITY ? 0.f : m[v]));
            l[v] += p;
            p_sm[kk * GT + head_of(v)] = p;
        }
        __syncwarp();
        // A block's products are summed before they are added to the output: the chain of additions into it
        // is as long as the item's blocks, not its keys.  Eight heads take the block in two turns
        // (registers).
#pragma unroll
        for (int g0 = 0; g0 < GT; g0 += GP) {
            if (g0 > 0) __syncwarp();
            float acc[GP][E];
#pragma unroll
            for (int k = 0; k < KB; ++k) {
                float p[GP], x[E];
                if constexpr (GP % 4 == 0) {
#pragma unroll
                    for (int g = 0; g < GP; g += 4) {
                        const float4 f = *reinterpret_cast<const float4 *>(p_sm + k * GT + g0 + g);
                        p[g] = f.x;
                        p[g + 1] = f.y;
                        p[g + 2] = f.z;
                        p[g + 3] = f.w;
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < GP; g += 2) {
                        const float2 f = *reinterpret_cast<const float2 *>(p_sm + k * GT + g0 + g);
                        p[g] = f.x;
                        p[g + 1] = f.y;
                    }
                }
                if constexpr (E == 4) {
                    const float4 f = lds_f4(Vs + k * ROW + lane * 16);
                    x[0] = f.x;
                    x[1] = f.y;
                    x[2] = f.z;
                    x[3] = f.w;
                } else {
                    const float2 f = lds_f2(Vs + k * ROW + lane * 8);
                    x[0] = f.x;
                    x[1] = f.y;
                }
#pragma unroll
                for (int g = 0; g < GP; ++g)
#pragma unroll
                    for (int e = 0; e < E; ++e) acc[g][e] = k ? fmaf(p[g], x[e], acc[g][e]) : p[g] * x[e];
            }
#pragma unroll
            for (int g = 0; g < GP; ++g)
#pragma unroll
                for (int e = 0; e < E; ++e) o[g0 + g][e] += acc[g][e];
        }
    }

    __device__ __forceinline__ void finish()
    {
#pragma unroll
        for (int v = 0; v < VPL; ++v)
#pragma unroll
            for (int o2 = 4; o2 <= 16; o2 <<= 1) l[v] += __shfl_xor_sync(0xffffffffu, l[v], o2);
        __syncwarp();  // the probabilities have been read
    }

    template <typename F> __device__ __forceinline__ void each_lse(int G, F f) const
    {
#pragma unroll
        for (int v = 0; v < VPL; ++v) {
            const int g = head_of(v);
            if (lane == lane_of(g) && g < G) f(g, m[v], l[v]);
        }
    }

    __device__ __forceinline__ void store(void *out, bool bf16, long qrow0, int G) const
    {
#pragma unroll
        for (int g = 0; g < GT; ++g) {
            const float lg = __shfl_sync(0xffffffffu, l[value_of(g)], lane_of(g));
            if (g < G) {
                const float inv = lg > 0.f ? 1.f / lg : 0.f;
#pragma unroll
                for (int e = 0; e < E; ++e) store_out(out, bf16, (qrow0 + g) * D + lane * E + e, o[g][e] * inv);
            }
        }
    }

    __device__ __forceinline__ void store_partial(float *po, int G) const
    {
#pragma unroll
        for (int g = 0; g < GT; ++g)
            if (g < G) {
                float *dst = po + (size_t)g * D + lane * E;
                if constexpr (E == 4) *reinterpret_cast<float4 *>(dst) = make_float4(o[g][0], o[g][1], o[g][2], o[g][3]);
                else *reinterpret_cast<float2 *>(dst) = make_float2(o[g][0], o[g][1]);
            }
    }
};

template <class Block>
__global__ void __launch_bounds__(kDecodeWarps * 32, 1)
    decode_stream(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV, DecodeArgs a)
{
    constexpr int D = Block::D, KB = Block::KB;
    using LY = RingLayout<D>;
    constexpr int NW = kDecodeWarps, S = kDecodeStages;
    constexpr int STAGE = LY::STAGE;
    constexpr int APP = Block::APP;  // 16-byte chunks of the appended K and V rows per lane
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[NW * S];  // ring stages of all warps (either partition)
    __shared__ int sm_scan[NW];
    __shared__ int sm_red[2 * NW];  // per warp: most blocks of a unit, units with keys
    __shared__ __align__(16) float sm_block[Block::SCRATCH > 0 ? NW * Block::SCRATCH : 1];  // the block consumer's
    const uint32_t raw0 = (uint32_t)__cvta_generic_to_shared(smem_raw);
    const uint32_t ring0 = (raw0 + 1023u) & ~1023u;
    int *sm_pre = reinterpret_cast<int *>(smem_raw + (ring0 - raw0) + LY::RING);  // [units + 1]
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int P = a.units;  // cache units
    if (Block::TENSOR_MAPS && tid == 0) {  // fetch both descriptors (kernel parameters) while the previous kernel drains
        prefetch_tensormap(&tmK);
        prefetch_tensormap(&tmV);
    }
    if (lane == 0) {
        for (int s2 = 0; s2 < S; ++s2) mbar_init((uint32_t)__cvta_generic_to_shared(&bars[wid * S + s2]), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        fence_async_shared();
    }
    __syncwarp();
    wait_prior_grid();  // lens, q and the new rows may come from the previous kernels
    const long long rs = ring_row(a);  // the ring row this launch writes (-1: none)

    // ---- plan: identical in every CTA (lens are not modified until every warp is done).
    // Each unit's keys form nb_u = ceil(le_u / KB) blocks; the blocks of all units are laid
    // end to end (prefix pb) and every working warp takes one contiguous range of equal
    // length, cut across unit boundaries (a stream-K split).  A unit cut between warps
    // leaves partial (max, sum, output) triples that its last piece merges.  Short units
    // (<= kMaxWholeBlocks blocks) are never cut: a range start inside one moves to the
    // unit's nearer end, since there a merge costs more than the imbalance it removes.
    int *pb = sm_pre;  // [units + 1] prefix of blocks
    const int seg = (P + blockDim.x - 1) / blockDim.x;
    const int u_lo = min(P, tid * seg), u_hi = min(P, u_lo + seg);
    // stage the lengths in the (still idle) ring memory with one coalesced sweep; the
    // plan below reads them from there (the ring is first written by TMA after the plan)
    int *len_sm = reinterpret_cast<int *>(smem_raw + (ring0 - raw0));
    for (int u0 = 0; u0 < P; u0 += 8 * (int)blockDim.x) {
        int Lr[8];  // all loads of the batch in flight before any store or error report
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int u = u0 + k * (int)blockDim.x + tid;
            Lr[k] = u < P ? __ldcg(a.lens + u) : 0;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int u = u0 + k * (int)blockDim.x + tid;
            if (u < P) {
                const bool ok = unit_ok(Lr[k], a.L_cap, a.append);
                if (!ok && blockIdx.x == 0)
                    raise_error(a.err, (a.append && Lr[k] == a.L_cap) ? ERR_ROOM : ERR_LEN);
                len_sm[u] = ok ? Lr[k] + a.append : 0;
            }
        }
    }
    __syncthreads();
    // While the plan is made (2 to 4 us) HBM would idle.  With many units most warps start at or near
    // a unit's first rows: each CTA sends its share of the units' first two blocks to L2 now (1792
    // units of 40 to 200 rows 32.7 -> 30.5 us, of 200 to 600 rows 78.2 -> 77.2 us; four blocks 31.8;
    // with fewer units than half the warps nothing changes).
    if (2 * P >= (int)gridDim.x * NW)
        for (int u = blockIdx.x + tid * gridDim.x; u < P; u += blockDim.x * gridDim.x) {
            const int rows = min(len_sm[u] - a.append, 2 * KB);  // rows in the cache
            if (rows <= 0) continue;
            const size_t off = (size_t)u * a.L_cap * Block::ROW;
            bulk_prefetch(static_cast<const char *>(a.K) + off, rows * Block::ROW);
            bulk_prefetch(static_cast<const char *>(a.V) + off, rows * Block::ROW);
        }
    {
        int my_b = 0, my_max = 0, my_ne = 0;
        for (int u = u_lo; u < u_hi; ++u) {
            const int nb = (len_sm[u] + KB - 1) / KB;
            my_b += nb;
            my_max = max(my_max, nb);
            my_ne += nb > 0;
        }
        int f = my_b;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int nf = __shfl_up_sync(0xffffffffu, f, o);
            if (lane >= o) f += nf;
        }
        my_max = __reduce_max_sync(0xffffffffu, (unsigned)my_max);
        my_ne = __reduce_add_sync(0xffffffffu, (unsigned)my_ne);
        if (lane == 31) sm_scan[wid] = f;
        if (lane == 0) {
            sm_red[wid] = my_max;
            sm_red[NW + wid] = my_ne;
        }
        __syncthreads();
        int rb = f - my_b;
        for (int w2 = 0; w2 < wid; ++w2) rb += sm_scan[w2];
        for (int u = u_lo; u < u_hi; ++u) {
            pb[u] = rb;
            rb += (len_sm[u] + KB - 1) / KB;
        }
        if (tid == blockDim.x - 1) pb[P] = rb;
    }
    __syncthreads();
    const int total_warps = gridDim.x * NW;
    int max_nb = 0, n_ne = 0;  // most blocks of one unit; units with keys
#pragma unroll
    for (int w2 = 0; w2 < NW; ++w2) {
        max_nb = max(max_nb, sm_red[w2]);
        n_ne += sm_red[NW + w2];
    }
    // Units of more than 8 query heads may run as two virtual units of half the heads over the same
    // rows (float32 always does): twice as many units keep more warps busy, their merges are half as
    // large, and the second read of a row mostly hits L2.  One pass for all heads is faster only with
    // many short units (few cuts) and many blocks per warp.  One pass : halves, us, 9 and 16 heads:
    // 1792 units of 225 to 300 rows 63 : 70 and 68 : 70, 896 of 375 to 500 51 : 55 and 57 : 57, of 600 to 800
    // 70 : 73 and 76 : 75; but 448 of 750 to 1000 57 : 51 and 65 : 53, of 2000 to 4100 142 : 128 (16 heads), 224
    // of 2250 to 3000 81 : 66 and 88 : 68, 64 of 6000 to 8000 91 : 58 and 96 : 62, 896 of 150 to 200 30 : 29 and
    // 30 : 29.
    const bool one_pass = P >= one_pass_units(total_warps) && pb[P] >= kOnePassBlocks * total_warps;
    const int hs = !Block::SPLIT ? 1 : (Block::ALWAYS ? 2 : (one_pass ? a.hs_min : a.hs_max));
    // Virtual unit u covers half u / P (of gv heads) of the cache unit u % P: all first halves come
    // first in the plan, then all second halves in the same order, so warps w and w + W/2 stream
    // the same rows at about the same time and the second read mostly hits L2.
    const int units = Block::SPLIT ? hs * P : P, GS = Block::SPLIT ? (a.G + hs - 1) / hs : a.G;
    auto cache_unit = [&](int u) { return Block::SPLIT && u >= P ? u - P : u; };
    auto head_part = [&](int u) { return Block::SPLIT && u >= P ? 1 : 0; };
    auto eff_len = [&](int u) {
        const int L = a.lens[cache_unit(u)];
        return unit_ok(L, a.L_cap, a.append) ? L + a.append : -1;
    };
    const int NB = (Block::SPLIT ? hs : 1) * pb[P];
    n_ne *= Block::SPLIT ? hs : 1;
    if (Block::SPLIT && hs == 2) {
        __syncthreads();  // pb[P] has been read
        for (int u = u_lo; u < u_hi; ++u) pb[P + u] = NB / 2 + pb[u];
        if (tid == blockDim.x - 1) pb[units] = NB;
        __syncthreads();
    }
    // Long work (at least kDeepBlocksPerWarp blocks per warp) runs on half the warps, each
    // with a ring twice as deep: more bytes in flight per warp keep HBM busier once every
    // warp has many blocks; short work keeps all warps for latency.  The CTA's ring is the
    // same either way (NW * S stages).
    // Fewer than half as many units as warps (with at least 8 blocks per warp) also
    // takes the deep partition: there the 8-warp split would cut every unit into many
    // pieces, whose merges cost more than the shallower rings save.
    // Not halves: their second read comes from L2, so warps wait less for data and more for each other
    // (448 units of 2000 to 4100 rows, 16 heads, 215 us on half the warps, 128 on all; 224 of 1500 to 2000 74
    // and 53).
    const bool deep = Block::DEEP && hs == 1 && GS <= 8 && (NB >= kDeepBlocksPerWarp * total_warps ||
                                      (NB >= 8 * total_warps && total_warps > 2 * units));
    // Only short units (none is ever cut): the contiguous deal below would leave some warps
    // two whole units where others have one.  Instead the units are sorted by blocks, most
    // first (ties by index, so every CTA builds the same order), and dealt in snake order:
    // warp w takes sorted units w, 2W-1-w, 2W+w, ... of W = min(warps, units with keys),
    // so a warp holding one of the longest units in a round holds one of the shortest in
    // the next.  The order replaces the block prefix in shared memory; units without keys
    // sort last.
    const bool snake = !deep && max_nb <= kMaxWholeBlocks;
    int *order = sm_pre;
    if (snake) {
        constexpr int NBK = kMaxWholeBlocks + 1;  // buckets: 16 - blocks, so most blocks first
        int *cnt = len_sm + ((P + 31) & ~31);  // [NBK][blockDim.x], also in the idle ring
        for (int k = 0; k < NBK; ++k) cnt[k * blockDim.x + tid] = 0;
        for (int u = u_lo; u < u_hi; ++u) cnt[(kMaxWholeBlocks - ((len_sm[u] + KB - 1) / KB)) * blockDim.x + tid] += Block::SPLIT ? hs : 1;
        __syncthreads();
        // exclusive scan of cnt in memory order (bucket-major, then thread): thread t takes
        // entries [NBK t, NBK (t + 1))
        int loc = 0;
        for (int k = 0; k < NBK; ++k) loc += cnt[tid * NBK + k];
        int f = loc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int nf = __shfl_up_sync(0xffffffffu, f, o);
            if (lane >= o) f += nf;
        }
        __syncthreads();  // every thread has read its entries (and NB, before the order overwrites pb)
        if (lane == 31) sm_scan[wid] = f;
        __syncthreads();
        int run = f - loc;
        for (int w2 = 0; w2 < wid; ++w2) run += sm_scan[w2];
        for (int k = 0; k < NBK; ++k) {
            const int c2 = cnt[tid * NBK + k];
            cnt[tid * NBK + k] = run;
            run += c2;
        }
        __syncthreads();
        // each thread places its own units, in index order, from its own column of cnt
        for (int u = u_lo; u < u_hi; ++u) {
            int &at = cnt[(kMaxWholeBlocks - ((len_sm[u] + KB - 1) / KB)) * blockDim.x + tid];
            order[at++] = u;
            if (Block::SPLIT && hs == 2) order[at++] = P + u;
        }
        __syncthreads();
    }
    bool aborted = false;
    // Working warps W: every one gets at least kMinBlocksPerWarp blocks (or all warps work), and no unit is
    // cut into too many pieces: one warp merges a unit's pieces one after another, each at about the cost
    // of (GS + 1) / 8 blocks.  With NB / W blocks per warp and max_nb * W / NB pieces of the longest unit, the
    // one time falls as the other grows; they are about equal at W^2 = 8 NB^2 / (max_nb (GS + 1)).  Up to
    // kCheapPieces pieces the merge costs less than the idle warps would.  us on all warps and so: 2 units
    // of 32000 rows, 7 heads 358 and 65; one such unit among 200 of 16 rows 372 and 75, among 15 of 900
    // rows 361 and 65.  Units of one length are cut into one number of pieces, unless that leaves warps idle that
    // have 8 blocks or more to do: then no warp has two pieces, of which each costs it a publication (some
    // 5 us: 8 units of 500 rows 20.8 on 45 warps, 18.2 on 64; 200 of 763 rows, 7 heads, 32.8 on 1216, 27.5 on
    // 1200; 224 units of 1500 rows, 44 blocks a warp, are bound by their bytes on either).
    const int all_warps = (deep ? NW / 2 : NW) * (int)gridDim.x;
    int W = max(1, min(all_warps, NB / kMinBlocksPerWarp));
    if (!snake) {  // (in floats: 64-bit products and divisions here cost a short call 0.2 to 0.5 us)
        const float fb = (float)NB;
        if ((float)max_nb * (float)W > kCheapPieces * fb)
            W = max(1, min(W, (int)(fb * rsqrtf(0.125f * (float)max_nb * (float)(GS + 1)))));
        if ((W < all_warps || NB < 8 * all_warps) && W >= n_ne && n_ne > 0 && NB - max_nb * n_ne == 0) W -= W % n_ne;
    }
    // the warp's items, by block consumer C
    auto run = [&](auto tag) {
    using C = typename decltype(tag)::type;
    constexpr int GM = C::GM;
    const int NWm = deep ? NW / 2 : NW, Sm = deep ? 2 * S : S;  // NWm * Sm == NW * S either way
    const uint32_t my_ring = ring0 + (uint32_t)wid * Sm * STAGE;
    const bool out_bf16 = a.out_bf16 != 0;
    auto wstart = [&](int w) { return (int)((long long)w * NB / W); };  // ideal first block of warp w
    auto owner = [&](int b) { return (int)(((long long)(b + 1) * W - 1) / NB); };  // ideal owner of block b

    // A piece: the part of unit u inside one warp's block range.  A unit cut between warps
    // wf .. wf+nsplit-1 keeps warp w's partial in slot 2w (the warp's first piece) or 2w+1
    // (its last piece): only those two pieces of a warp can be partial.  Only long units
    // are cut, and no range start moves inside a long unit, so there the ideal owners hold.
    struct Item {
        int u, pu, hp, ub, wf, nsplit, slot, slot0, le, k0, k1, Lapp, nblk;  // pu, hp: cache unit, head part
    };
    auto last_le = [](const int *pre, int units_, int d) {  // largest u with pre[u] <= d
        int lo = 0, hi = units_ - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (pre[mid] <= d) lo = mid; else hi = mid - 1;
        }
        return lo;
    };
    auto snap = [&](int b) {  // a range start inside a short unit moves to its nearer end
        if (b >= NB) return NB;
        const int u = last_le(pb, units, b);
        const int ub = pb[u], ue = pb[u + 1];
        if (ue - ub > kMaxWholeBlocks) return b;
        return b - ub <= ue - b ? ub : ue;
    };
    // static deal interleaved across CTAs (warp wid of every CTA before warp wid+1 of
    // any): with fewer working warps than warps the work still spreads over all SMs
    const int gw = wid * (int)gridDim.x + (int)blockIdx.x;
    const bool working = gw < W && !snake;
    const int b_end = working ? snap(wstart(gw + 1)) : 0;
    int b_next = working ? snap(wstart(gw)) : 0;
    int eu = gw;  // next unit this warp checks for emptiness (empty units: no blocks)
    const int Ws = min(NW * (int)gridDim.x, n_ne);  // snake deal: warps with units
    int sk = 0, spos = gw < Ws ? gw : n_ne;          // round and sorted position of the next unit
    auto next_item = [&]() {
        Item it;
        it.nblk = -1;  // no item
        if (snake) {
            if (spos < n_ne) {
                const int u = order[spos];
                const int le_raw = eff_len(u);
                it.u = u;
                it.pu = cache_unit(u);
                it.hp = head_part(u);
                it.ub = 0;
                it.le = le_raw >= 0 ? le_raw : 0;
                it.Lapp = (le_raw >= 0 && a.append) ? it.le - 1 : -1;
                it.k0 = 0;
                it.k1 = it.le;
                it.nblk = (it.le + KB - 1) / KB;
                it.wf = gw;
                it.nsplit = 1;
                it.slot = it.slot0 = 0;
                ++sk;
                spos = sk * Ws + ((sk & 1) ? Ws - 1 - gw : gw);
                return it;
            }
            while (n_ne + eu < units) {  // units without keys: zero output, lse = -inf
                const int u = order[n_ne + eu];
                eu += total_warps;
                it.u = u;
                it.pu = cache_unit(u);
                it.hp = head_part(u);
                it.ub = 0;
                it.le = 0;
                it.Lapp = -1;
                it.k0 = it.k1 = 0;
                it.nblk = 0;
                it.wf = 0;
                it.nsplit = 1;
                it.slot = it.slot0 = 0;
                return it;
            }
            return it;
        }
        if (b_next < b_end) {
            const int u = last_le(pb, units, b_next);  // the nonempty unit holding block b_next
            const int ub = pb[u], ue = pb[u + 1];
            const int bend = min(b_end, ue);
            const int le_raw = eff_len(u);
            it.u = u;
            it.pu = cache_unit(u);
            it.hp = head_part(u);
            it.ub = ub;
            it.le = le_raw >= 0 ? le_raw : 0;
            it.Lapp = (le_raw >= 0 && a.append) ? it.le - 1 : -1;
            it.k0 = (b_next - ub) * KB;
            it.k1 = min((bend - ub) * KB, it.le);
            it.nblk = bend - b_next;
            if (ue - ub <= kMaxWholeBlocks) {  // a short unit: always whole
                it.wf = gw;
                it.nsplit = 1;
                it.slot = it.slot0 = 0;
            } else {
                it.wf = owner(ub);
                it.nsplit = owner(ue - 1) - it.wf + 1;
                it.slot0 = 2 * it.wf + (snap(wstart(it.wf)) < ub ? 1 : 0);  // warp wf's slot
                it.slot = gw == it.wf ? it.slot0 : 2 * gw;
            }
            b_next = bend;
            return it;
        }
        while (eu < units) {  // units without keys: zero output, lse = -inf
            const int u = eu;
            eu += total_warps;
            if (pb[u + 1] == pb[u]) {
                const int le_raw = eff_len(u);
                it.u = u;
                it.pu = cache_unit(u);
                it.hp = head_part(u);
                it.ub = pb[u];
                it.le = 0;
                it.Lapp = -1;
                it.k0 = it.k1 = 0;
                it.nblk = 0;
                it.wf = 0;
                it.nsplit = 1;
                it.slot = it.slot0 = 0;
                (void)le_raw;
                return it;
            }
        }
        return it;
    };

    C blk(lane, C::SCRATCH > 0 ? sm_block + wid * C::SCRATCH : nullptr);
    auto load_q = [&](const Item &it) {
        const long qrow = (long)(it.pu / a.Hkv) * a.Hq + (long)(it.pu % a.Hkv) * a.G + it.hp * GS;
        blk.load_q(a.q, qrow, min(GS, a.G - it.hp * GS));
    };

    // K and V rows are read once per launch: evict them first, so they do not displace the
    // queries, the outputs, the partials or the next kernels' inputs from L2 (a medium cache,
    // 1792 units of 200-400 rows, went from 62.1 to 56.6 us; the 7B-class launch 1.5% faster)
    const uint64_t kv_policy = l2_evict_first_policy();
    // ---- block stream: lane 0 keeps up to S blocks in flight, running from the current
    // item into the next one (grabbed one item ahead) so no refill bubble opens between
    // items; the warp consumes blocks in issue order.
    uint32_t issued = 0, consumed = 0;
    uint32_t p_slot = 0, c_slot = 0, c_par = 0;  // ring slot of the next issue / next wait, wait phase
    Item cur = next_item();
    Item nxt;
    nxt.nblk = -1;  // looked up below, after the first copies are out
    Item pit = cur;  // item the producer is issuing from
    int pblk = 0;
    bool p_on_next = false;
    auto can_issue = [&]() {
        if (pblk < pit.nblk) return true;
        if (!p_on_next && nxt.nblk > 0) {
            pit = nxt;
            pblk = 0;
            p_on_next = true;
            return true;
        }
        return false;
    };
    auto issue = [&]() {
        const uint32_t slot = p_slot;
        if (lane == 0) {
            const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&bars[wid * Sm + slot]);
            const uint32_t dst = my_ring + slot * STAGE;
            fence_async_shared();
            const int k = pit.k0 + KB * pblk;  // first key; the appended row is not in the cache yet
            Block::load(dst, bar, &tmK, &tmV, a, pit.pu, k, min(KB, (pit.Lapp >= 0 ? pit.Lapp : pit.le) - k), kv_policy);
        }
        ++pblk;
        ++issued;
        if (++p_slot == (uint32_t)Sm) p_slot = 0;
    };
    // the first piece's copies go out before the next piece is looked up (that lookup
    // reads a length from global memory)
    __syncwarp();
    while (issued < (uint32_t)Sm && pblk < pit.nblk) issue();
    if (cur.nblk >= 0) load_q(cur);  // the queries of the next item to start
    nxt = cur.nblk >= 0 ? next_item() : cur;
    // the launch's queries into the window ring (row rs of every query head's `slots`
    // rows): each warp copies an equal share of 16-byte chunks while its first copies
    // are in flight
    if (a.qring != nullptr && rs >= 0) {
        constexpr int CH = Block::ROW / 16;  // 16-byte chunks of a query row
        const long long n16 = a.nq_rows * CH;
        const int tw = (int)gridDim.x * NW, me = (int)blockIdx.x * NW + wid;
        const long long per = (n16 + tw - 1) / tw;
        const long long c0 = min(n16, (long long)me * per), c1 = min(n16, c0 + per);
        const uint4 *src = reinterpret_cast<const uint4 *>(a.q);
        uint4 *dst = reinterpret_cast<uint4 *>(a.qring);
        for (long long cb = c0; cb < c1; cb += 32 * 8) {
            uint4 v[8];  // all loads in flight before the stores
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const long long c = cb + 32 * k + lane;
                if (c < c1) v[k] = __ldcg(src + c);
            }
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const long long c = cb + 32 * k + lane;
                if (c < c1) dst[(c / CH * a.slots + rs) * CH + c % CH] = v[k];
            }
        }
    }

    while (cur.nblk >= 0) {
        const int u = cur.u, k0 = cur.k0, k1 = cur.k1, Lapp = cur.Lapp;
        const int nsplit = cur.nsplit, item = cur.slot, wf = cur.wf, slot0 = cur.slot0;  // partial slots
        const int pu = cur.pu;  // the cache unit
        const long lb = pu / a.Hkv;
        const int h = pu % a.Hkv;
        const int G = min(GS, a.G - cur.hp * GS);
        const long qrow0 = lb * a.Hq + (long)h * a.G + cur.hp * GS;
        // this lane's 16-byte chunks of the appended rows (K's chunks, then V's), loaded now so that
        // neither the stage patch nor the cache write below waits on global memory
        constexpr int CPR = Block::ROW / 16;
        uint4 app[APP];
        const bool has_app = Lapp >= k0 && Lapp < k1;
#pragma unroll
        for (int i = 0; i < APP; ++i) {
            const int p = lane + 32 * i;
            app[i] = make_uint4(0, 0, 0, 0);
            if (has_app && p < 2 * CPR)
                app[i] = reinterpret_cast<const uint4 *>(p < CPR ? a.k_new : a.v_new)[(long)pu * CPR + p % CPR];
        }

        // start this item's copies before the wait on its query registers below
        __syncwarp();
        while (issued - consumed < (uint32_t)Sm && can_issue()) issue();
        blk.start();
        if (nxt.nblk >= 0) load_q(nxt);  // the next item's queries load while this one streams

        for (int bi = 0; bi < cur.nblk; ++bi) {
            __syncwarp();
            while (issued - consumed < (uint32_t)Sm && can_issue()) issue();
            const uint32_t slot = c_slot, parity = c_par;
            const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&bars[wid * Sm + slot]);
            if (!mbar_wait_bounded(bar, parity, kSpinLimit)) {  // a copy never landed: report, drain, stop
                if (lane == 0) raise_error(a.err, ERR_INTERNAL);
                for (uint32_t q2 = consumed + 1; q2 < issued; ++q2)
                    mbar_wait_bounded((uint32_t)__cvta_generic_to_shared(&bars[wid * Sm + q2 % Sm]), (q2 / Sm) & 1u,
                                      kSpinLimit);
                aborted = true;
                break;
            }
            const int kb = k0 + KB * bi;
            const uint32_t Ks = my_ring + slot * STAGE, Vs = Ks + STAGE / 2;
            // patch the stage: zero V rows past the item (K rows there are masked), and
            // put the appended row (not yet in the cache) in place
            if (kb + KB > k1 || (Lapp >= kb && Lapp < kb + KB)) {
                const int zr = max(k1 - kb, 0);
                for (int p = lane; p < (KB - zr) * CPR; p += 32)
                    sts_u4(Vs + Block::chunk(zr + p / CPR, p % CPR), make_uint4(0, 0, 0, 0));
                if (Lapp >= kb && Lapp < kb + KB) {
#pragma unroll
                    for (int i = 0; i < APP; ++i) {
                        const int p = lane + 32 * i;
                        if (p < 2 * CPR) sts_u4((p < CPR ? Ks : Vs) + Block::chunk(Lapp - kb, p % CPR), app[i]);
                    }
                }
                __syncwarp();
            }
            blk.consume(Ks, Vs, kb, k1, a.c2);
            ++consumed;
            if (++c_slot == (uint32_t)Sm) {
                c_slot = 0;
                c_par ^= 1u;
            }
        }
        if (aborted) break;

        blk.finish();

        // the warp that covers the appended index writes the new row into the cache
        if (has_app && cur.hp == 0) {
#pragma unroll
            for (int i = 0; i < APP; ++i) {
                const int p = lane + 32 * i;
                if (p < 2 * CPR)
                    reinterpret_cast<uint4 *>(p < CPR ? a.K : a.V)[((long)pu * a.L_cap + Lapp) * CPR + p % CPR] = app[i];
            }
        }

        if (nsplit == 1) {
            blk.store(a.out, out_bf16, qrow0, G);
            blk.each_lse(G, [&](int q, float m, float l) {
                put_lse(a, rs, qrow0 + q, l > 0.f ? (m + log2f(l)) * kLn2 : -INFINITY);
            });
        } else {
            blk.store_partial(a.part_o + (size_t)item * GS * D, G);
            blk.each_lse(G, [&](int q, float m, float l) {
                reinterpret_cast<float2 *>(a.part_ml)[(size_t)item * GS + q] = make_float2(m, l);
            });
            // publish: the warp barrier orders every lane's partial writes before lane 0's
            // release; the last arriver's acquire (and the barrier after it) orders its reads
            __syncwarp();
            int old = 0;
            if (lane == 0) old = atom_add_acq_rel(&a.counters[2 + u], 1);
            old = __shfl_sync(0xffffffffu, old, 0);
            __syncwarp();
            if (old == nsplit - 1) {  // last item of this unit: merge the partials
                if (lane == 0) a.counters[2 + u] = 0;  // every piece has counted: clear for the next launch
                // pass 1: per-query-head maxima, lanes over splits (independent loads)
                float Mq[GM];
#pragma unroll
                for (int qq = 0; qq < GM; ++qq) Mq[qq] = -INFINITY;
                for (int sb = 0; sb < nsplit; sb += 32) {
                    const int s2 = sb + lane;
                    if (s2 < nsplit) {
#pragma unroll
                        for (int qq = 0; qq < GM; ++qq)
                            if (qq < G)
                                Mq[qq] = fmaxf(Mq[qq], __ldcg(a.part_ml + ((size_t)(s2 ? 2 * (wf + s2) : slot0) * GS + qq) * 2));
                    }
                }
#pragma unroll
                for (int qq = 0; qq < GM; ++qq) Mq[qq] = warp_max(Mq[qq]);
                // pass 2: every lane owns 4 head-dim elements of all G heads; one sweep over
                // the splits with all of a split's loads issued together
                constexpr int PER = D / 32;
                float acc[GM][PER], Lq[GM];
#pragma unroll
                for (int qq = 0; qq < GM; ++qq) {
                    Lq[qq] = 0.f;
#pragma unroll
                    for (int e = 0; e < PER; ++e) acc[qq][e] = 0.f;
                }
#pragma unroll 2
                for (int s2 = 0; s2 < nsplit; ++s2) {
                    const size_t it0 = (size_t)(s2 ? 2 * (wf + s2) : slot0) * GS;
#pragma unroll
                    for (int qq = 0; qq < GM; ++qq) {
                        if (qq < G && Mq[qq] != -INFINITY) {
                            const float2 ml = __ldcg(reinterpret_cast<const float2 *>(a.part_ml) + it0 + qq);
                            const float wt = fast_exp2(ml.x - Mq[qq]);
                            Lq[qq] += ml.y * wt;
                            const float *src = a.part_o + (it0 + qq) * D + lane * PER;
                            if constexpr (PER == 4) {
                                const float4 ov = __ldcg(reinterpret_cast<const float4 *>(src));
                                acc[qq][0] += ov.x * wt;
                                acc[qq][1] += ov.y * wt;
                                acc[qq][2] += ov.z * wt;
                                acc[qq][3] += ov.w * wt;
                            } else {
#pragma unroll
                                for (int e = 0; e < PER; ++e) acc[qq][e] += __ldcg(src + e) * wt;
                            }
                        }
                    }
                }
#pragma unroll
                for (int qq = 0; qq < GM; ++qq) {
                    if (qq < G) {
                        const float inv = Lq[qq] > 0.f ? 1.f / Lq[qq] : 0.f;
#pragma unroll
                        for (int e = 0; e < PER; ++e)
                            store_out(a.out, out_bf16, (qrow0 + qq) * D + lane * PER + e,
                                                     acc[qq][e] * inv);
                        if (lane == 0)
                            put_lse(a, rs, qrow0 + qq, Lq[qq] > 0.f ? (Mq[qq] + log2f(Lq[qq])) * kLn2 : -INFINITY);
                    }
                }
            }
        }
        // advance: the producer may already be streaming the next item's blocks
        cur = nxt;
        nxt = cur.nblk >= 0 ? next_item() : cur;
        if (p_on_next) {
            p_on_next = false;
        } else {
            pit = cur;
            pblk = 0;
        }
    }
    };
    if constexpr (std::is_same_v<Block, typename Block::Half>) {  // one consumer
        run(Tag<Block>{});
    } else if (GS > 8) {
        run(Tag<Block>{});
    } else {
        run(Tag<typename Block::Half>{});
    }

    // Every warp, stopped early or not, counts itself done with one 64-bit add on the
    // pair counters[0..1]: +1 on counters[1] (warps done) and, for a stopped warp, +1 on
    // counters[0] (warps stopped), so the value the add returns tells the last warp of
    // every stop before it, with no further read.  The last one has every other warp
    // behind it: it advances the lengths (every plan has been read by then) and clears
    // the counters, so a launch leaves the workspace's counters zero as it found them,
    // also after a stop.
    unsigned long long dc = 0;
    const bool stopped = __shfl_sync(0xffffffffu, aborted, 0);
    __syncwarp();
    if (lane == 0)
        dc = atom_add_acq_rel_u64(reinterpret_cast<unsigned long long *>(a.counters),
                                  (1ull << 32) | (stopped ? 1ull : 0ull));
    dc = __shfl_sync(0xffffffffu, dc, 0);
    __syncwarp();
    if ((int)(dc >> 32) == total_warps - 1) {
        const bool any_stop = stopped || (uint32_t)dc != 0u;
        if (any_stop) {  // tickets of units whose pieces stopped early may still count
            for (int u = lane; u < units; u += 32) a.counters[2 + u] = 0;
        } else if (a.append) {
            // 16 independent loads per lane in flight before any store, of 4 lengths each
            // when lens is 16-byte aligned: one L2 round trip for up to 2048 units
            constexpr int BATCH = 16;
            const int cu = P;  // cache units
            const int n4 = (reinterpret_cast<uintptr_t>(a.lens) & 15u) == 0 ? cu / 4 : 0;
            int4 *l4 = reinterpret_cast<int4 *>(a.lens);
            for (int i0 = 0; i0 < n4; i0 += 32 * BATCH) {
                int4 L[BATCH];
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {
                    const int i = i0 + 32 * k + lane;
                    L[k] = i < n4 ? __ldcg(l4 + i) : make_int4(-1, -1, -1, -1);
                }
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {
                    const int i = i0 + 32 * k + lane;
                    if (i < n4) {
                        int4 v = L[k];
                        v.x += unit_ok(v.x, a.L_cap, a.append) ? 1 : 0;
                        v.y += unit_ok(v.y, a.L_cap, a.append) ? 1 : 0;
                        v.z += unit_ok(v.z, a.L_cap, a.append) ? 1 : 0;
                        v.w += unit_ok(v.w, a.L_cap, a.append) ? 1 : 0;
                        l4[i] = v;
                    }
                }
            }
            for (int u0 = 4 * n4; u0 < cu; u0 += 32 * BATCH) {  // the rest (or all) one length at a time
                int L[BATCH];
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {
                    const int u = u0 + 32 * k + lane;
                    L[k] = u < cu ? __ldcg(a.lens + u) : -1;
                }
#pragma unroll
                for (int k = 0; k < BATCH; ++k) {
                    const int u = u0 + 32 * k + lane;
                    if (u < cu && unit_ok(L[k], a.L_cap, a.append)) a.lens[u] = L[k] + 1;
                }
            }
        }
        __syncwarp();
        if (lane == 0) {
            *reinterpret_cast<unsigned long long *>(a.counters) = 0ull;
            if (rs >= 0 && a.advance) *a.slot = (rs + 1) % a.slots;  // every warp has read the row by now
        }
    }
}

// The launch's queries into the window ring after the SIMT decode: chunk c (16 bytes)
// of query row c / ch goes to row *slot of that head's `slots` rows.
__global__ void qring_copy(const uint4 *__restrict__ q, uint4 *__restrict__ qring, long long n16, int ch, int slots,
                           const long long *slot)
{
    const long long s = *slot;
    if (s < 0 || s >= slots) return;  // the decode has reported the slot
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n16; c += (long long)gridDim.x * blockDim.x)
        qring[(c / ch * slots + s) * ch + c % ch] = q[c];
}

// The ring slot's advance after the SIMT decode (its CTAs have no last-warp step).
__global__ void ring_advance(long long *slot, int slots)
{
    const long long s = *slot;
    if (s >= 0 && s < slots) *slot = (s + 1) % slots;
}

// ---------------------------------------------------------------- host side
// [rows, d] bf16 view of a cache tensor, 16-row x 64-column boxes, 128-byte swizzle.
static bool encode_cache_map(CUtensorMap *map, const void *base, unsigned long long rows, int d)
{
    return encode_bf16_2d(map, base, rows, d, 64, 16);
}

typedef void (*DecodeKernel)(CUtensorMap, CUtensorMap, DecodeArgs);

// float32 kernel for up to gt (2, 4, 6 or 8) query heads per virtual unit.
template <int D> static DecodeKernel f32_kernel(int gt)
{
    switch (gt) {
    case 2: return decode_stream<F32Block<D, 2>>;
    case 4: return decode_stream<F32Block<D, 4>>;
    case 6: return decode_stream<F32Block<D, 6>>;
    default: return decode_stream<F32Block<D, 8>>;
    }
}

// bf16 kernel: up to 8 query heads per unit, or up to 16, of which `halves` makes two units.
template <int D> static DecodeKernel bf16_kernel(bool wide, bool halves)
{
    if (!wide) return decode_stream<Bf16Block<D, 1>>;
    return halves ? decode_stream<Bf16Block<D, 1, 2>> : decode_stream<Bf16Block<D, 2>>;
}

cudaError_t launch_decode(const reco_kv &kv, const void *q, const void *k_new, const void *v_new,
                          int32_t *lens, float scale, void *out, reco_dtype out_dtype, float *lse,
                          const DecodeWs &ws, unsigned *err, cudaStream_t s, float *ring, int slots,
                          long long *slot, void *qring)
{
    DecodeArgs a;
    a.K = kv.k;
    a.V = kv.v;
    a.q = q;
    a.k_new = k_new;
    a.v_new = v_new;
    a.lens = lens;
    a.out = out;
    a.lse = lse;
    a.counters = ws.counters;
    a.part_ml = ws.part_ml;
    a.part_o = ws.part_o;
    a.units = kv.n_layers * kv.B * kv.H_kv;
    a.Hq = kv.H_q;
    a.Hkv = kv.H_kv;
    a.G = kv.H_q / kv.H_kv;
    a.L_cap = kv.L_cap;
    a.append = (k_new && v_new) ? 1 : 0;
    a.out_bf16 = out_dtype == RECO_BF16 ? 1 : 0;
    a.c2 = scale * kLog2e;
    a.err = err;
    a.ring = ring;
    a.slot = slot;
    a.slots = slots;
    a.nq = (long long)kv.n_layers * kv.B * kv.H_q;
    a.qring = ring ? qring : nullptr;
    a.nq_rows = a.nq;
    a.advance = 1;
    const bool f32 = kv.dtype == RECO_F32;
    // virtual units per unit: float32 units of more than 8 heads run as two of half as many; bf16
    // ones may (the kernel decides from the lengths), as long as one plan holds all units twice
    const int hs = f32 && a.G > 8 ? 2 : 1;
    a.hs_min = hs;
    DecodeKernel fn;
    if (f32) {
        const int gt = a.G > 6 ? 8 : (a.G + 1) / 2 * 2;  // (halves of more than 8 heads: by the widest)
        fn = kv.d == 64 ? f32_kernel<64>(gt) : f32_kernel<128>(gt);
    } else {
        // With more than 8 heads: calls that run as halves in any case, as few units or a cache that cannot
        // hold 24 blocks a warp tell, take the kernel of one consumer (64 units of 6000 to 8000 rows, 16
        // heads, 62 us against 69 in the kernel that may choose, 448 of 750 to 1000 53 against 58).
        const int warps = kDecodeWarps * device_sm_count();
        const bool halves = a.G > 8 && 2LL * std::min<long long>(a.units, kMaxTmaUnits) <= kMaxTmaUnits &&
                            (a.units < one_pass_units(warps) || (long long)a.units * ((kv.L_cap + 15) / 16) < 24LL * warps);
        fn = kv.d == 64 ? bf16_kernel<64>(a.G > 8, halves) : bf16_kernel<128>(a.G > 8, halves);
    }
    // More units than one plan holds in shared memory run as consecutive launches over
    // contiguous unit ranges (every unit is independent): each part gets its own K/V, q,
    // output, lens and ring pointers, and only the last part advances the ring slot.
    const long long part_units = (f32 ? kMaxF32Units : kMaxTmaUnits) / hs;  // cache units per launch
    // bf16 rows are addressed by tensor-map coordinates
    if (f32 || (unsigned long long)std::min<long long>(a.units, part_units) * kv.L_cap < (1ull << 31)) {
        const size_t row_b = (size_t)kv.d * (f32 ? 4 : 2);  // cache and query rows
        const size_t out_b = (size_t)kv.d * (out_dtype == RECO_BF16 ? 2 : 4);
        for (long long u0 = 0; u0 < a.units; u0 += part_units) {
            const long long cu = std::min(part_units, (long long)a.units - u0);
            const long long q0 = u0 * a.G;  // first query head of the part
            const unsigned long long rows = (unsigned long long)cu * kv.L_cap;
            CUtensorMap mk = {}, mv = {};
            const char *kb = static_cast<const char *>(kv.k) + (size_t)u0 * kv.L_cap * row_b;
            const char *vb = static_cast<const char *>(kv.v) + (size_t)u0 * kv.L_cap * row_b;
            if (!f32 && (!encode_cache_map(&mk, kb, rows, kv.d) || !encode_cache_map(&mv, vb, rows, kv.d))) {
                if (u0 == 0) break;  // the SIMT path below takes the whole call
                return cudaErrorInvalidValue;
            }
            DecodeArgs at = a;  // this part
            at.units = (int)cu;
            at.hs_max = a.G > 8 && 2 * cu <= (f32 ? kMaxF32Units : kMaxTmaUnits) ? 2 : hs;
            at.K = const_cast<char *>(kb);
            at.V = const_cast<char *>(vb);
            at.q = static_cast<const char *>(q) + (size_t)q0 * row_b;
            at.k_new = k_new ? static_cast<const char *>(k_new) + (size_t)u0 * row_b : nullptr;
            at.v_new = v_new ? static_cast<const char *>(v_new) + (size_t)u0 * row_b : nullptr;
            at.lens = lens + u0;
            at.out = static_cast<char *>(out) + (size_t)q0 * out_b;
            at.lse = lse ? lse + q0 : nullptr;
            at.ring = ring ? ring + q0 : nullptr;  // ring rows keep their full stride nq
            at.qring = a.qring ? static_cast<char *>(a.qring) + (size_t)q0 * slots * row_b : nullptr;
            at.nq_rows = cu * a.G;
            at.advance = u0 + cu >= a.units ? 1 : 0;
            // the counters are zero on entry (zero-filled workspace) and every launch leaves them so
            const int plan = at.units * at.hs_max;
            const size_t smem = kv.d == 64 ? ring_smem_bytes<64>(plan) : ring_smem_bytes<128>(plan);
            cudaError_t e = allow_smem((const void *)fn, (int)smem);
            if (e != cudaSuccess) return e;
            // two partial slots per warp of the grid
            const int grid = std::min(device_sm_count(), ws.part_slots / (2 * kDecodeWarps));
            e = launch_pdl(fn, dim3(grid), dim3(kDecodeWarps * 32), smem, s, mk, mv, at);
            if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
            if (u0 + cu >= a.units) return cudaSuccess;
        }
    }
    // bf16 caches that no tensor map covers
    const unsigned grid = (unsigned)a.units;
    if (kv.d == 64) decode_simt<__nv_bfloat16, 64><<<grid, 128, 0, s>>>(a);
    else decode_simt<__nv_bfloat16, 128><<<grid, 128, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !ring) return e;
    if (a.qring) {
        const int ch = kv.d * 2 / 16;
        const long long n16 = a.nq * ch;
        const unsigned blocks = (unsigned)std::min<long long>((n16 + 255) / 256, 4LL * device_sm_count());
        qring_copy<<<blocks, 256, 0, s>>>(reinterpret_cast<const uint4 *>(q), reinterpret_cast<uint4 *>(a.qring), n16,
                                          ch, slots, slot);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    ring_advance<<<1, 1, 0, s>>>(slot, slots);
    return cudaGetLastError();
}

}  // namespace reco
