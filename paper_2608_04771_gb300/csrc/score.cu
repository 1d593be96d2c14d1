// score.cu -- Eq. 2 (Sec. 3.2, attention-guided selection): per-KV-head cache scores.
//
// s_j = (1/G) sum_g sum_t softmax_j(scale * q_{g,t} . k_j), window query t at position
// L-w+t seeing keys j <= L-w+t, then a max-pool over the candidate range [0, L-w).
//
// A softmax row needs its max and normaliser over ALL keys before any column can be
// summed, so the scores take two passes over K:
//   pass 1  per (unit, key chunk): per-row running max / sum in the log2 domain
//   combine per (unit, row): merge the chunk partials -> b_r = m_r + log2 Z_r
//   pass 2  per (unit, key tile): column sums  sum_r 2^(c*l_rj - b_r) / G
//   pool    per (unit, key): max over the clipped window
// This file holds the SIMT passes used for float32 caches (and any shape the tensor-
// core passes do not cover), the combine and pool kernels, and the launcher;
// score_tc.cu holds the bf16 tensor-core (tcgen05) passes.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "score_plan.cuh"

namespace reco {

bool score_tc_supported(const reco_kv &kv, int w);

// Partials of a window row in the workspace.  Tensor-core shapes: up to two per chunk (a chunk's
// key tiles are split between two epilogue groups).  Others: one per tile of keys, so that the
// tiles of a short call spread over the SMs.
static int score_row_parts(const reco_kv &kv, int w)
{
    return score_tc_supported(kv, w) ? 2 * ((kv.L_cap + kScoreChunk - 1) / kScoreChunk) : (kv.L_cap + kTile - 1) / kTile;
}

// Tiles per partial on plain FMAs (a tensor-core shape gets there only without tensor maps).
static int simt_part_tiles(const reco_kv &kv, int w) { return score_tc_supported(kv, w) ? kScoreChunk / kTile : 1; }

ScoreWs score_ws_layout(const reco_kv &kv, int w, void *base)
{
    size_t units = (size_t)kv.n_layers * kv.B * kv.H_kv;
    size_t R = (size_t)(kv.H_q / kv.H_kv) * w;
    char *p = (char *)base;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *r = p ? p + off : nullptr;
        off += align256(bytes);
        return r;
    };
    ScoreWs ws;
    const size_t parts = score_row_parts(kv, w);  // per row
    ws.part_m = (float *)take(units * parts * R * 4);
    ws.part_z = (float *)take(units * parts * R * 4);
    ws.rowb = (float *)take(units * R * 4);
    ws.raw = (float *)take(units * (size_t)kv.L_cap * 4);
    ws.ulist = (int32_t *)take(units * 4);
    ws.ucount = (int32_t *)take(4);
    ws.bytes = off;
    return ws;
}

// ---------------------------------------------------------------- passes on plain FMAs
// float32 caches (and bf16 shapes the tensor-core passes do not cover): every product and sum in
// float32.  Both passes are register-tiled: a CTA holds a tile of 128 keys in shared memory and
// takes the unit's window rows 64 at a time, each of its 256 threads computing a 4 x 8 block of
// logits from float4 reads along d (rows ty + 16 i, keys tx + 16 j; the row stride of D + 4 floats
// keeps the reads of a quarter-warp on different banks).  The CTAs, two per SM so that one loads
// while the other multiplies, share the call's tiles as the plan deals them.
//
// The FMA issue bounds it: a thread's 128 FMAs per four elements of d come with 12 shared-memory
// reads (paired FMAs, which halve the instructions, bring nothing).  Both passes over 64 units of about
// 3500 keys, d 128, 192 window rows: 2400 -> 536 us replayed from a graph (42 TFLOP/s, 52% of the FMA
// rate; 564 to 620 us as calls among others) from one key or row per thread, one read per four FMAs
// and 2048 keys a CTA.
constexpr int kSimtRows = 64, kSimtThreads = 256;

template <int D> struct SimtSmem {
    static constexpr int LD = D + 4;  // floats per row
    static constexpr size_t BYTES = (size_t)(kTile + kSimtRows) * LD * sizeof(float);
};

// `rows` rows of D elements from src into dst (float32, LD apart), of which `valid` exist; zeros
// stand for the others.
template <typename T, int D>
__device__ __forceinline__ void simt_load(float *dst, const T *__restrict__ src, int rows, int valid)
{
    constexpr int C = D / 4;  // groups of four elements per row
#pragma unroll 8
    for (int e = threadIdx.x; e < rows * C; e += kSimtThreads) {
        const int r = e / C, c = 4 * (e % C);
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < valid) {
            if constexpr (sizeof(T) == 4) {
                v = __ldg(reinterpret_cast<const float4 *>(src + (long)r * D + c));
            } else {
                const uint2 x = __ldg(reinterpret_cast<const uint2 *>(src + (long)r * D + c));
                const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x.x));
                const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x.y));
                v = make_float4(lo.x, lo.y, hi.x, hi.y);
            }
        }
        *reinterpret_cast<float4 *>(dst + r * SimtSmem<D>::LD + c) = v;
    }
}

// s[i][j] = row ty + 16 i of Qs . row tx + 16 j of Ks
template <int D> __device__ __forceinline__ void simt_logits(const float *Qs, const float *Ks, float (&s)[4][8])
{
    constexpr int LD = SimtSmem<D>::LD;
    const float *q = Qs + (threadIdx.x >> 4) * LD, *k = Ks + (threadIdx.x & 15) * LD;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) s[i][j] = 0.f;
#pragma unroll 4
    for (int c = 0; c < D; c += 4) {
        float4 a[4], b[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4 *>(q + 16 * i * LD + c);
#pragma unroll
        for (int j = 0; j < 8; ++j) b[j] = *reinterpret_cast<const float4 *>(k + 16 * j * LD + c);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                s[i][j] = fmaf(a[i].x, b[j].x, s[i][j]);
                s[i][j] = fmaf(a[i].y, b[j].y, s[i][j]);
                s[i][j] = fmaf(a[i].z, b[j].z, s[i][j]);
                s[i][j] = fmaf(a[i].w, b[j].w, s[i][j]);
            }
    }
}

// Pass 1: one (max, sum) partial per window row and part_tiles tiles of keys (one CTA's, one after
// another: the row's thread adds each to the partial).
template <typename T, int D>
__global__ void __launch_bounds__(kSimtThreads, 2) score_rowstats_simt(
    const T *__restrict__ q_win, const T *__restrict__ K, const int32_t *__restrict__ lens, ScoreMask mask, int w, int G,
    int Hq, int Hkv, int L_cap, int R, int n_parts, int part_tiles, int units, float c2, float *__restrict__ part_m,
    float *__restrict__ part_z, unsigned *err)
{
    extern __shared__ __align__(16) float smem[];
    float *Ks = smem, *Qs = smem + kTile * SimtSmem<D>::LD;
    __shared__ TilePlan plan;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    wait_prior_grid();  // lens, the queries and the cache may come from the previous kernels
    for (int skip = 0, n_runs = 1; skip < n_runs; skip += kPlanRuns) {
        n_runs = plan_runs<1>(plan, lens, mask, w, L_cap, units, false, part_tiles * kTile, skip, nullptr, nullptr, err);
        for (int e = 0; e < min(kPlanRuns, n_runs - skip); ++e) {
            const TileRun run = plan.run[e];
            const T *q = q_win + ((long)(run.u / Hkv) * Hq + (long)(run.u % Hkv) * G) * w * D;
            for (int t = run.t0; t < run.t0 + run.nt; ++t) {
                const int j0 = t * kTile;
                for (int r0 = 0; r0 < R; r0 += kSimtRows) {
                    __syncthreads();  // the tiles before these have been read
                    if (r0 == 0) simt_load<T, D>(Ks, K + ((long)run.u * L_cap + j0) * D, kTile, run.L - j0);
                    simt_load<T, D>(Qs, q + (long)r0 * D, kSimtRows, R - r0);
                    __syncthreads();
                    float s[4][8];
                    simt_logits<D>(Qs, Ks, s);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = r0 + ty + 16 * i;
                        const int last = min(run.L - 1, run.L - w + r % w);  // the last key this row sees
                        float m = -INFINITY, z = 0.f;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            s[i][j] = j0 + tx + 16 * j <= last ? s[i][j] * c2 : -INFINITY;
                            m = fmaxf(m, s[i][j]);
                        }
#pragma unroll
                        for (int o = 8; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                        const float base = m == -INFINITY ? 0.f : m;
#pragma unroll
                        for (int j = 0; j < 8; ++j) z += fast_exp2(s[i][j] - base);
#pragma unroll
                        for (int o = 8; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
                        if (tx == 0 && r < R) {
                            const size_t o = ((size_t)run.u * n_parts + t / part_tiles) * R + r;
                            if (t % part_tiles) lse_merge(m, z, part_m[o], part_z[o]);
                            part_m[o] = m;
                            part_z[o] = z;
                        }
                    }
                }
            }
        }
    }
}

// Merge the partials of each row (`per` of them for each part_keys keys, laid out
// [unit][n_parts][R]) into b_r = m_r + log2(Z_r).
__global__ void score_combine(const int32_t *__restrict__ lens, ScoreMask mask, int w, int L_cap, int R,
                              int n_parts, int part_keys, int per, const float *__restrict__ part_m,
                              const float *__restrict__ part_z, float *__restrict__ rowb, long units)
{
    wait_prior_grid();  // the partials come from pass 1
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= units * R) return;
    long u = i / R;
    int r = (int)(i % R);
    int L = lens[u];
    if (L < w || L > L_cap || mask.skip(u, L, w, L_cap)) return;
    const int used = ((L + part_keys - 1) / part_keys) * per;
    float m = -INFINITY, z = 0.f;
    const size_t o0 = (size_t)u * n_parts * R + r;
    constexpr int U = 8;  // partials in flight: their max, then one exponential each
    for (int c0 = 0; c0 < used; c0 += U) {
        float pm[U], pz[U], mn = m;
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const bool in = c0 + k < used;
            const size_t o = o0 + (size_t)(c0 + k) * R;
            pm[k] = in ? part_m[o] : -INFINITY;
            pz[k] = in ? part_z[o] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < U; ++k) mn = fmaxf(mn, pm[k]);
        if (mn == -INFINITY) continue;
        z *= fast_exp2(m - mn);
#pragma unroll
        for (int k = 0; k < U; ++k) z = fmaf(pz[k], fast_exp2(pm[k] - mn), z);
        m = mn;
    }
    rowb[i] = m + log2f(z);
}

// Row normalisers from log-sum-exps the decode already produced (Eq. 2 with one pass over
// K).  Window row (g, t) is query head g of the token at position L - w + t; when that
// token was decoded the cache held exactly the keys j <= L - w + t that Eq. 2's causal
// mask gives the row, so the decode's natural-log normaliser lse of that query head is
// the row's: b_r = lse * log2(e).  row_lse is [w][rows_q] (rows_q = layers * B * H_q,
// query heads in q order).  A non-finite normaliser raises ERR_NORM and leaves the row's
// normaliser at +inf, so the row adds nothing to the scores.  The tensor-core pass 2
// computes the same b_r itself where it loads a row's normaliser; this kernel serves
// the SIMT pass.
__global__ void score_rowb_from_lse(const int32_t *__restrict__ lens, ScoreMask mask, int w, int L_cap, int R, int G,
                                    int Hq, int Hkv, long rows_q, const float *__restrict__ row_lse,
                                    float *__restrict__ rowb, long units, unsigned *err)
{
    wait_prior_grid();  // lens and the ring rows may come from the previous kernels
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= units * R) return;
    const long u = i / R;
    const int r = (int)(i % R);
    const int L = lens[u];
    if (L < w || L > L_cap) {  // no other pass of this call reports it
        if (r == 0) raise_error(err, ERR_LEN);
        return;
    }
    if (mask.skip(u, L, w, L_cap)) return;
    const int g = r / w, t = r % w;
    const long qi = (u / Hkv) * Hq + (u % Hkv) * G + g;
    const float lse = row_lse[(long)t * rows_q + qi];
    if (!isfinite(lse)) {
        raise_error(err, ERR_NORM);
        rowb[i] = INFINITY;
        return;
    }
    rowb[i] = lse * kLog2e;
}

// lse ring of 2 * slots rows: rows *slot and *slot + slots both get lse[0:n] (the second
// half mirrors the first, so the rows of any `slots` consecutive pushes are contiguous),
// then *slot = (*slot + 1) % slots.  One block: every thread reads the slot before thread
// 0 advances it.
__global__ void __launch_bounds__(1024) lse_push_kernel(const float *__restrict__ lse, long n, float *__restrict__ ring,
                                                        int slots, long long *slot, unsigned *err)
{
    wait_prior_grid();  // lse (and the slot) may come from the previous kernels
    __shared__ long long s0;
    if (threadIdx.x == 0) s0 = *slot;
    __syncthreads();
    const long long s = s0;
    if (s < 0 || s >= slots) {
        if (threadIdx.x == 0) raise_error(err, ERR_INTERNAL);
        return;
    }
    float *dst = ring + s * n, *mir = ring + (s + slots) * n;
    // four independent loads in flight per thread before their stores
    constexpr int U = 4;
    if (n % 4 == 0 &&
        ((reinterpret_cast<uintptr_t>(lse) | reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(mir)) & 15u) == 0) {
        const float4 *src4 = reinterpret_cast<const float4 *>(lse);
        float4 *dst4 = reinterpret_cast<float4 *>(dst), *mir4 = reinterpret_cast<float4 *>(mir);
        const long n4 = n / 4;
        for (long i0 = threadIdx.x; i0 < n4; i0 += (long)U * blockDim.x) {
            float4 v[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const long i = i0 + (long)k * blockDim.x;
                if (i < n4) v[k] = src4[i];
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const long i = i0 + (long)k * blockDim.x;
                if (i < n4) {
                    dst4[i] = v[k];
                    mir4[i] = v[k];
                }
            }
        }
    } else {
        for (long i0 = threadIdx.x; i0 < n; i0 += (long)U * blockDim.x) {
            float v[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const long i = i0 + (long)k * blockDim.x;
                if (i < n) v[k] = lse[i];
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const long i = i0 + (long)k * blockDim.x;
                if (i < n) {
                    dst[i] = v[k];
                    mir[i] = v[k];
                }
            }
        }
    }
    if (threadIdx.x == 0) *slot = (s + 1) % slots;
}

// Pass 2: every thread's column sums over its rows, added over the row threads at the tile's end.
// PAD: the rows end inside a tile of 64 (a kernel of its own: testing the rows costs whole tiles 1%,
// and spares 32-row calls 1% of their exponentials).
template <typename T, int D, bool PAD>
__global__ void __launch_bounds__(kSimtThreads, 2) score_colsum_simt(
    const T *__restrict__ q_win, const T *__restrict__ K, const int32_t *__restrict__ lens, ScoreMask mask, int w, int G,
    int Hq, int Hkv, int L_cap, int R, int units, float c2, const float *__restrict__ rowb, float *__restrict__ raw,
    int32_t *ulist, int32_t *ucount)
{
    extern __shared__ __align__(16) float smem[];
    float *Ks = smem, *Qs = smem + kTile * SimtSmem<D>::LD;
    __shared__ TilePlan plan;
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float invG = 1.f / (float)G;
    wait_prior_grid();  // lens, the normalisers, the queries and the cache may come from the previous kernels
    for (int skip = 0, n_runs = 1; skip < n_runs; skip += kPlanRuns) {
        n_runs = plan_runs<1>(plan, lens, mask, w, L_cap, units, true, kTile, skip, ulist, ucount, nullptr);
        for (int e = 0; e < min(kPlanRuns, n_runs - skip); ++e) {
            const TileRun run = plan.run[e];
            const int nc = run.L - w;
            const T *q = q_win + ((long)(run.u / Hkv) * Hq + (long)(run.u % Hkv) * G) * w * D;
            for (int t = run.t0; t < run.t0 + run.nt; ++t) {
                const int j0 = t * kTile;
                float sum[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int r0 = 0; r0 < R; r0 += kSimtRows) {
                    float b[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int r = r0 + ty + 16 * i;
                        b[i] = !PAD || r < R ? rowb[(long)run.u * R + r] : 0.f;
                    }
                    __syncthreads();  // the tiles before these have been read
                    if (r0 == 0) simt_load<T, D>(Ks, K + ((long)run.u * L_cap + j0) * D, kTile, nc - j0);
                    simt_load<T, D>(Qs, q + (long)r0 * D, kSimtRows, R - r0);
                    __syncthreads();
                    float s[4][8];
                    simt_logits<D>(Qs, Ks, s);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        // a padding row adds nothing, and its logit with an infinite key is NaN
                        if (PAD && r0 + ty + 16 * i >= R) break;
#pragma unroll
                        for (int j = 0; j < 8; ++j) sum[j] += fast_exp2(fmaf(s[i][j], c2, -b[i]));
                    }
                }
                __syncthreads();  // Qs has been read: the warps' sums go there
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    sum[j] += __shfl_xor_sync(0xffffffffu, sum[j], 16);
                    if (lane < 16) Qs[wid * kTile + tx + 16 * j] = sum[j];
                }
                __syncthreads();
                if (threadIdx.x < kTile && j0 + (int)threadIdx.x < nc) {
                    float a = 0.f;
#pragma unroll
                    for (int k = 0; k < kSimtThreads / 32; ++k) a += Qs[k * kTile + threadIdx.x];
                    raw[(long)run.u * L_cap + j0 + threadIdx.x] = a * invG;
                }
            }
        }
    }
}

// Max-pool over the clipped window [j - pool/2, j + pool/2] within [0, L-w).  A CTA pools
// kPoolTile scores of a unit from a shared-memory copy of them and their halo; scores outside the
// range are NaN there, which fmaxf passes over, so that no window needs clipping.  What bounds it
// is latency (length, scores, barrier, results), so a thread keeps 16 scores in flight: 7B-class
// cache, 14.2 M scores, took 55 us with one load per window entry.  Windows wider than the halo read global memory.
constexpr int kPoolTile = 4096, kPoolHalo = 64, kPoolThreads = 256;

__device__ __forceinline__ void pool_tile(const float *__restrict__ rp, int j0, int nc, int half,
                                          float *__restrict__ out, bool vec, float *sm)
{
    constexpr int Q = kPoolTile / kPoolThreads / 4;  // groups of four consecutive scores per thread
    const int n = min(kPoolTile, nc - j0);
    // at most a score per thread: straight from global memory, the window's loads in flight together (no
    // shared memory, no barrier: 0.2 of 7.4 us for one pass over 4 units of 120 keys)
    if (n <= kPoolThreads && half <= 4) {
        const int j = j0 + (int)threadIdx.x;
        if ((int)threadIdx.x < n) {
            float m = __int_as_float(0x7fc00000);
#pragma unroll
            for (int o = -4; o <= 4; ++o)
                if (o >= -half && o <= half && j + o >= 0 && j + o < nc) m = fmaxf(m, __ldcg(rp + j + o));
            out[j] = m;
        }
        return;
    }
    if (half > kPoolHalo) {
        for (int t = threadIdx.x; t < n; t += kPoolThreads) {
            const int j = j0 + t, lo = max(0, j - half), hi = min(nc - 1, j + half);
            float m = rp[lo];
            for (int i = lo + 1; i <= hi; ++i) m = fmaxf(m, rp[i]);
            out[j] = m;
        }
        return;
    }
    const float none = __int_as_float(0x7fc00000);
    float *c = sm + kPoolHalo;  // c[t] = score j0 + t
    if (vec) {                  // rows of whole, aligned groups of four (the group at nc stays inside the row)
        float4 v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int t = 4 * (threadIdx.x + q * kPoolThreads);
            v[q] = t < n ? __ldcg(reinterpret_cast<const float4 *>(rp + j0 + t)) : make_float4(none, none, none, none);
        }
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int t = 4 * (threadIdx.x + q * kPoolThreads);
            if (t + 1 >= n) v[q].y = none;
            if (t + 2 >= n) v[q].z = none;
            if (t + 3 >= n) v[q].w = none;
            *reinterpret_cast<float4 *>(c + t) = v[q];
        }
    } else {
        float v[4 * Q];
#pragma unroll
        for (int q = 0; q < 4 * Q; ++q) {
            const int t = threadIdx.x + q * kPoolThreads;
            v[q] = t < n ? __ldcg(rp + j0 + t) : none;
        }
#pragma unroll
        for (int q = 0; q < 4 * Q; ++q) c[threadIdx.x + q * kPoolThreads] = v[q];
    }
    if (threadIdx.x < 2 * kPoolHalo) {
        const int t = threadIdx.x < kPoolHalo ? (int)threadIdx.x - kPoolHalo : kPoolTile + (int)threadIdx.x - kPoolHalo;
        const int j = j0 + t;
        c[t] = j >= 0 && j < nc && t >= -half && t < kPoolTile + half ? __ldcg(rp + j) : none;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int t = 4 * (threadIdx.x + q * kPoolThreads);
        if (t >= n) break;
        float m[4];
        if (half <= 4) {
            float x[12];  // scores t - 4 .. t + 7
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const float4 f = *reinterpret_cast<const float4 *>(c + t - 4 + 4 * i);
                x[4 * i] = f.x;
                x[4 * i + 1] = f.y;
                x[4 * i + 2] = f.z;
                x[4 * i + 3] = f.w;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                m[k] = x[4 + k];
#pragma unroll
                for (int o = 1; o <= 4; ++o)
                    if (o <= half) m[k] = fmaxf(m[k], fmaxf(x[4 + k - o], x[4 + k + o]));
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) m[k] = none;
            for (int i = -half; i < half + 4; ++i) {
                const float x = c[t + i];
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (i >= k - half && i <= k + half) m[k] = fmaxf(m[k], x);
            }
        }
        if (vec && t + 4 <= n) {
            *reinterpret_cast<float4 *>(out + j0 + t) = make_float4(m[0], m[1], m[2], m[3]);
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (t + k < n) out[j0 + t + k] = m[k];
        }
    }
    __syncthreads();
}

// Whether a unit's rows of raw and scores are whole, aligned groups of four.
__device__ __forceinline__ bool pool_vec(const float *raw, const float *scores, int L_cap)
{
    return (L_cap & 3) == 0 && ((reinterpret_cast<uintptr_t>(raw) | reinterpret_cast<uintptr_t>(scores)) & 15u) == 0;
}

// The pool over the units of a masked call's list only: CTAs (blockIdx.x: a tile of scores)
// walk the list, so the units left out cost no CTAs.
__global__ void __launch_bounds__(kPoolThreads) score_pool_list(const float *__restrict__ raw, const int32_t *__restrict__ lens,
                                                       const int32_t *__restrict__ ulist,
                                                       const int32_t *__restrict__ ucount, int w, int L_cap, int pool,
                                                       float *__restrict__ scores)
{
    __shared__ __align__(16) float sm[kPoolTile + 2 * kPoolHalo];
    wait_prior_grid();  // the raw scores and the list come from the previous kernels
    const int n = *ucount;
    for (int k = blockIdx.y; k < n; k += gridDim.y) {
        const long u = ulist[k];
        const int L = lens[u], j0 = blockIdx.x * kPoolTile;
        if (L < w || L > L_cap || j0 >= L - w) continue;
        pool_tile(raw + u * L_cap, j0, L - w, pool / 2, scores + u * L_cap, pool_vec(raw, scores, L_cap), sm);
    }
}

__global__ void __launch_bounds__(kPoolThreads) score_pool(const float *__restrict__ raw, const int32_t *__restrict__ lens,
                                                  ScoreMask mask, int w, int L_cap, int pool,
                                                  float *__restrict__ scores)
{
    __shared__ __align__(16) float sm[kPoolTile + 2 * kPoolHalo];
    wait_prior_grid();  // the raw scores come from the previous kernel
    const long u = blockIdx.y;
    const int L = lens[u], j0 = blockIdx.x * kPoolTile;
    if (L < w || L > L_cap || mask.skip(u, L, w, L_cap) || j0 >= L - w) return;
    pool_tile(raw + u * L_cap, j0, L - w, pool / 2, scores + u * L_cap, pool_vec(raw, scores, L_cap), sm);
}

cudaError_t launch_score_tc_pass1(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask,
                                  int w, float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool *used);
// row_lse (or nullptr: ws.rowb) gives pass 2 its row normalisers: the decode's lse, read
// where each row's normaliser is loaded.
// A masked call's pass 2 also lists the units it scored in ws.ulist / ws.ucount.
cudaError_t launch_score_tc_pass2(const reco_kv &kv, const void *q_win, const int32_t *lens, const ScoreMask &mask,
                                  int w, float c2, const ScoreWs &ws, const float *row_lse, unsigned *err,
                                  cudaStream_t s, bool *used);
int score_tc_pass1_groups(int R);

// CTAs of a column-sum pass: one per SM on the tensor cores, two on plain FMAs.
static long colsum_ctas(bool tc) { return (tc ? 1L : 2L) * device_sm_count(); }

// Passes on plain FMAs; with pass1 false the row normalisers are already in ws.rowb.  A masked
// call's pass 2 also lists the units it scored in ws.ulist / ws.ucount.
template <typename T, int D>
static cudaError_t score_simt(const reco_kv &kv, const T *q_win, const int32_t *lens, ScoreMask mask, int w,
                              float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool pass1 = true)
{
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const int G = kv.H_q / kv.H_kv, R = G * w;
    const long tiles = units * ((kv.L_cap + kTile - 1) / kTile);
    const dim3 grid((unsigned)std::min(tiles, colsum_ctas(false))), block(kSimtThreads);
    constexpr size_t smem = SimtSmem<D>::BYTES;
    const T *K = (const T *)kv.k;
    cudaError_t e = cudaSuccess;
    if (pass1) {
        const int n_parts = score_row_parts(kv, w), part_tiles = simt_part_tiles(kv, w);
        e = allow_smem((const void *)score_rowstats_simt<T, D>, (int)smem);
        if (e != cudaSuccess) return e;
        e = launch_pdl(score_rowstats_simt<T, D>, grid, block, smem, s, q_win, K, lens, mask, w, G, kv.H_q, kv.H_kv,
                       kv.L_cap, R, n_parts, part_tiles, (int)units, c2, ws.part_m, ws.part_z, err);
        if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
        e = launch_pdl(score_combine, dim3((unsigned)((units * R + 255) / 256)), dim3(256), 0, s, lens, mask, w,
                       kv.L_cap, R, n_parts, part_tiles * kTile, 1, (const float *)ws.part_m, (const float *)ws.part_z, ws.rowb,
                       units);
        if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
    }
    auto colsum = R % kSimtRows ? score_colsum_simt<T, D, true> : score_colsum_simt<T, D, false>;
    e = allow_smem((const void *)colsum, (int)smem);
    if (e != cudaSuccess) return e;
    e = launch_pdl(colsum, grid, block, smem, s, q_win, K, lens, mask, w, G, kv.H_q, kv.H_kv, kv.L_cap,
                   R, (int)units, c2, (const float *)ws.rowb, ws.raw, mask.keep ? ws.ulist : nullptr,
                   mask.keep ? ws.ucount : nullptr);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Largest R*D (and R more) the calls outside the tensor-core passes accept: the shapes that fitted an
// earlier kernel, which held all of a unit's window queries in shared memory.  These passes need no
// limit; it stays as the interface's, with which callers choose their windows.
constexpr size_t kSimtMaxQ = 200 * 1024 / 4;

bool score_shape_supported(const reco_kv &kv, int w)
{
    size_t R = (size_t)(kv.H_q / kv.H_kv) * w;
    if (score_tc_supported(kv, w)) return true;
    return (kv.d == 64 || kv.d == 128) && (R * kv.d + R) <= kSimtMaxQ;
}

static cudaError_t score_simt_any(const reco_kv &kv, const void *q_win, const int32_t *lens, ScoreMask mask, int w,
                                  float c2, const ScoreWs &ws, unsigned *err, cudaStream_t s, bool pass1)
{
    if (kv.dtype == RECO_F32)
        return kv.d == 64 ? score_simt<float, 64>(kv, (const float *)q_win, lens, mask, w, c2, ws, err, s, pass1)
                          : score_simt<float, 128>(kv, (const float *)q_win, lens, mask, w, c2, ws, err, s, pass1);
    return kv.d == 64
               ? score_simt<__nv_bfloat16, 64>(kv, (const __nv_bfloat16 *)q_win, lens, mask, w, c2, ws, err, s, pass1)
               : score_simt<__nv_bfloat16, 128>(kv, (const __nv_bfloat16 *)q_win, lens, mask, w, c2, ws, err, s,
                                                pass1);
}

// Max-pooling of the raw scores into `scores`: over the unit list where the column sums (on the tensor
// cores, or not) built one, which a masked call's do unless every item has its CTA; else one CTA per
// (unit, tile of scores).
static cudaError_t launch_pool(const reco_kv &kv, const int32_t *lens, ScoreMask mask, bool tc, int w, int pool,
                               float *scores, const ScoreWs &ws, cudaStream_t s)
{
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const unsigned chunks = (unsigned)((kv.L_cap + kPoolTile - 1) / kPoolTile);
    if (mask.keep != nullptr && plan_items(units, kv.L_cap, kTile) > colsum_ctas(tc)) {
        const long walkers = std::max(1L, 8L * device_sm_count() / (long)chunks);
        const unsigned ys = (unsigned)std::min(units, std::min(walkers, 65535L));
        cudaError_t e = launch_pdl(score_pool_list, dim3(chunks, ys), dim3(kPoolThreads), 0, s, (const float *)ws.raw, lens,
                                   (const int32_t *)ws.ulist, (const int32_t *)ws.ucount, w, kv.L_cap, pool, scores);
        if (e != cudaSuccess) return e;
    } else {
        cudaError_t e = launch_pdl(score_pool, dim3(chunks, (unsigned)units), dim3(kPoolThreads), 0, s, (const float *)ws.raw, lens,
                                   mask, w, kv.L_cap, pool, scores);
        if (e != cudaSuccess) return e;
    }
    return cudaGetLastError();
}

cudaError_t launch_score(const reco_kv &kv, const void *q_win, const int32_t *lens, const int32_t *keep, int w,
                         int pool, float scale, float *scores, const ScoreWs &ws, unsigned *err, cudaStream_t s)
{
    const float c2 = scale * kLog2e;
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const ScoreMask mask{keep, kv.B, kv.H_kv};
    cudaError_t e = cudaSuccess;
    bool used_tc = false;
    const bool tc = kv.dtype == RECO_BF16 && score_tc_supported(kv, w);
    if (tc) {
        // tensor-core passes: pass 1 -> combine -> pass 2
        e = launch_score_tc_pass1(kv, q_win, lens, mask, w, c2, ws, err, s, &used_tc);
        if (e != cudaSuccess) return e;
        if (used_tc) {
            const int R = (kv.H_q / kv.H_kv) * w;
            const int nch = (kv.L_cap + kScoreChunk - 1) / kScoreChunk;
            e = launch_pdl(score_combine, dim3((unsigned)((units * R + 255) / 256)), dim3(256), 0, s, lens, mask, w,
                           kv.L_cap, R, nch * score_tc_pass1_groups(R), kScoreChunk, score_tc_pass1_groups(R),
                           (const float *)ws.part_m, (const float *)ws.part_z, ws.rowb, units);
            if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
            bool used2 = false;
            e = launch_score_tc_pass2(kv, q_win, lens, mask, w, c2, ws, nullptr, err, s, &used2);
            if (e != cudaSuccess) return e;
            if (!used2) return cudaErrorNotSupported;
        }
    }
    if (!used_tc) {
        e = score_simt_any(kv, q_win, lens, mask, w, c2, ws, err, s, true);
        if (e != cudaSuccess) return e;
    }
    return launch_pool(kv, lens, mask, used_tc, w, pool, scores, ws, s);
}

cudaError_t launch_lse_push(const float *lse, long n, float *ring, int slots, long long *slot, unsigned *err,
                            cudaStream_t s)
{
    cudaError_t e = launch_pdl(lse_push_kernel, dim3(1), dim3(1024), 0, s, lse, n, ring, slots, slot, err);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Row *index of a [rows][n16] array of 16-byte chunks into dst, for captured step loops
// whose input row is chosen on the device: a grid of a few CTAs per SM, eight independent
// 16-byte loads per thread in flight before its stores.
__global__ void __launch_bounds__(256) copy_row_kernel(const uint4 *__restrict__ src, long long rows, long long n16,
                                                     const long long *__restrict__ index, uint4 *__restrict__ dst,
                                                     unsigned *err)
{
    wait_prior_grid();  // the index (and the destination's readers) belong to earlier kernels
    const long long r = *index;
    if (r < 0 || r >= rows) {
        if (blockIdx.x == 0 && threadIdx.x == 0) raise_error(err, ERR_INTERNAL);
        return;
    }
    const uint4 *row = src + r * n16;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < n16; i0 += 8 * stride) {
        uint4 v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long i = i0 + k * stride;
            if (i < n16) v[k] = ld_stream_u4(row + i);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const long long i = i0 + k * stride;
            if (i < n16) dst[i] = v[k];
        }
    }
}

cudaError_t launch_copy_row(const void *src, long long rows, long long row_bytes, const long long *index, void *dst,
                            unsigned *err, cudaStream_t s)
{
    const long long n16 = row_bytes / 16;
    const long long want = (n16 + 256LL * 8 - 1) / (256LL * 8);
    const unsigned grid = (unsigned)std::max(1LL, std::min(want, 4LL * device_sm_count()));
    cudaError_t e = launch_pdl(copy_row_kernel, dim3(grid), dim3(256), 0, s, reinterpret_cast<const uint4 *>(src), rows,
                               n16, index, reinterpret_cast<uint4 *>(dst), err);
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_score_lse(const reco_kv &kv, const void *q_win, const int32_t *lens, const int32_t *keep,
                             const float *row_lse, int w, int pool, float scale, float *scores, const ScoreWs &ws,
                             unsigned *err, cudaStream_t s)
{
    const float c2 = scale * kLog2e;
    const long units = (long)kv.n_layers * kv.B * kv.H_kv;
    const ScoreMask mask{keep, kv.B, kv.H_kv};
    const int G = kv.H_q / kv.H_kv, R = G * w;
    const long rows_q = (long)kv.n_layers * kv.B * kv.H_q;
    const bool tc = kv.dtype == RECO_BF16 && score_tc_supported(kv, w);
    cudaError_t e;
    bool used = false;
    if (tc) {  // the tensor-core pass reads each row's normaliser from row_lse itself
        e = launch_score_tc_pass2(kv, q_win, lens, mask, w, c2, ws, row_lse, err, s, &used);
        if (e != cudaSuccess) return e;
    }
    if (!used) {  // the SIMT pass takes them from ws.rowb
        e = launch_pdl(score_rowb_from_lse, dim3((unsigned)((units * R + 255) / 256)), dim3(256), 0, s, lens, mask, w,
                       kv.L_cap, R, G, kv.H_q, kv.H_kv, rows_q, row_lse, ws.rowb, units, err);
        if (e != cudaSuccess || (e = cudaGetLastError()) != cudaSuccess) return e;
        e = score_simt_any(kv, q_win, lens, mask, w, c2, ws, err, s, false);
        if (e != cudaSuccess) return e;
    }
    return launch_pool(kv, lens, mask, used, w, pool, scores, ws, s);
}

}  // namespace reco
