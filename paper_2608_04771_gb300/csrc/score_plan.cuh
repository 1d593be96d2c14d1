// score_plan.cuh -- how the scoring passes share a call's work between their CTAs.
#pragma once
#include "common.cuh"
#include "internal.h"

namespace reco {

// Every CTA builds the same plan from lens (and keep): the prefix, in unit order, of the
// units' work items (an item is `item_keys` keys of one unit), cut into one equal contiguous
// range per CTA.  A CTA keeps only the runs of its own range: run = tiles [t0, t0 + nt) of
// unit u.  Units without work (skipped, empty, out of range) take no run and no items, so
// ragged lengths and masked calls leave the CTAs evenly loaded.  A CTA whose range covers
// more than kPlanRuns units plans and runs it in rounds of kPlanRuns.
//
// The plan costs a small call more than its tiles do, so what it waits for is kept short: a call
// whose every possible item has a CTA of its own is not planned at all (an item's CTA reads one
// length; 4 units of 120 keys, 224 window rows, one pass 9.2 -> 7.4 us with this and the columns split four ways), the warps' totals are added by reductions, the
// ranges need no 64-bit division, and a thread keeps its units' lengths in registers between the
// sweeps where they are few (the trace's boundary, 1792 units: 18.2 -> 16.8 us).
constexpr int kPlanRuns = 256;
constexpr int kTile = 128;  // keys per tile, both passes

struct TileRun {
    int u, L, t0, nt;
};

struct TilePlan {
    TileRun run[kPlanRuns];
    int items[32], units[32];  // per warp: items and units with work
    int first, n;              // rank of the range's first unit among those with work; runs of the range
};

// Items that the units' rows can hold.
__host__ __device__ __forceinline__ long long plan_items(long long units, int L_cap, int item_keys)
{
    return units * ((L_cap + item_keys - 1) / item_keys);
}

template <int HELD>
__device__ __forceinline__ int plan_runs(TilePlan &pl, const int32_t *__restrict__ lens, const ScoreMask &mask, int w,
                                         int L_cap, int units, bool candidates_only, int item_keys, int skip,
                                         int32_t *ulist, int32_t *ucount, unsigned *err_len);

// The plan out of line, for kernels whose main loops suffer from the inlined one (long tensor-core
// calls: one pass over 8 layers of the 32B-class heads 643 -> 627 us).
static __device__ __noinline__ int plan_runs_call(TilePlan &pl, const int32_t *__restrict__ lens, const ScoreMask &mask,
                                                  int w, int L_cap, int units, bool candidates_only, int item_keys,
                                                  int skip, int32_t *ulist, int32_t *ucount, unsigned *err_len)
{
    return plan_runs<1>(pl, lens, mask, w, L_cap, units, candidates_only, item_keys, skip, ulist, ucount, err_len);
}

// Runs skip .. skip + kPlanRuns of this CTA's range into pl.run; returns the range's runs.
// Given ulist, CTA 0 also lists every unit with work (ascending) and their count, unless every item has
// its CTA (then a masked call has few units at most); given err_len, lengths out of range are
// reported, also of units that the mask leaves out.  HELD > 1: a thread keeps the lengths of its units,
// up to HELD of them (calls with more plan out of line); HELD = 1: of its only unit, or reads them
// again.  All threads of the CTA call it; it ends with a CTA barrier and keeps the plans of
// consecutive rounds apart.
template <int HELD>
__device__ __forceinline__ int plan_runs(TilePlan &pl, const int32_t *__restrict__ lens, const ScoreMask &mask, int w,
                                         int L_cap, int units, bool candidates_only, int item_keys, int skip,
                                         int32_t *ulist, int32_t *ucount, unsigned *err_len)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    if (plan_items(units, L_cap, item_keys) == gridDim.x) {
        const int per_unit = (L_cap + item_keys - 1) / item_keys;
        const int u = (int)blockIdx.x / per_unit, c = (int)blockIdx.x - u * per_unit;
        const int L = lens[u];
        int k = 0;  // keys of the item
        if (L < w || L > L_cap) {
            if (err_len != nullptr && c == 0 && tid == 0) raise_error(err_len, ERR_LEN);
        } else if (mask.keep == nullptr || mask.keep[(u / mask.Hkv) % mask.B] < L) {
            k = min(item_keys, (candidates_only ? L - w : L) - c * item_keys);
        }
        if (k <= 0) return 0;
        if (tid == 0) pl.run[0] = TileRun{u, L, c * (item_keys / kTile), (k + kTile - 1) / kTile};
        __syncthreads();
        return 1;
    }
    if (HELD > 1 && units > HELD * nt)
        return plan_runs_call(pl, lens, mask, w, L_cap, units, candidates_only, item_keys, skip, ulist, ucount, err_len);
    const int seg = (units + nt - 1) / nt;
    const int u_lo = min(units, tid * seg), u_hi = min(units, u_lo + seg);
    bool bad = false;  // a length out of range: reported after the sweep, whose loads an atomic would hold back
    auto keys_of = [&](int u, int &L) {
        L = lens[u];
        const int kp = mask.keep != nullptr ? mask.keep[(u / mask.Hkv) % mask.B] : 0;  // (its load does not wait for the length)
        if (L < w || L > L_cap) {
            bad = true;
            return 0;
        }
        if (mask.keep != nullptr && kp >= L) return 0;
        return candidates_only ? L - w : L;
    };
    int my_i = 0, my_n = 0, Lh[HELD] = {}, kh[HELD] = {};
    if constexpr (HELD > 1) {
#pragma unroll
        for (int i = 0; i < HELD; ++i)
            if (u_lo + i < u_hi) kh[i] = keys_of(u_lo + i, Lh[i]);
#pragma unroll
        for (int i = 0; i < HELD; ++i) {
            my_i += (kh[i] + item_keys - 1) / item_keys;
            my_n += kh[i] > 0;
        }
    } else {
#pragma unroll 4
        for (int u = u_lo; u < u_hi; ++u) {
            int L;
            const int k = keys_of(u, L);
            Lh[0] = L;
            kh[0] = k;
            my_i += (k + item_keys - 1) / item_keys;
            my_n += k > 0;
        }
    }
    if (bad && err_len != nullptr && blockIdx.x == 0 && skip == 0) raise_error(err_len, ERR_LEN);
    int fi = my_i, fn = my_n;  // inclusive scans within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int a = __shfl_up_sync(0xffffffffu, fi, o), b = __shfl_up_sync(0xffffffffu, fn, o);
        if (lane >= o) {
            fi += a;
            fn += b;
        }
    }
    __syncthreads();  // the previous round's runs have been walked
    if (lane == 31) {
        pl.items[wid] = fi;
        pl.units[wid] = fn;
    }
    if (tid == 0) pl.n = 0;
    __syncthreads();
    const int wi = lane < nw ? pl.items[lane] : 0, wn = lane < nw ? pl.units[lane] : 0;
    const int tot_i = __reduce_add_sync(0xffffffffu, wi), tot_n = __reduce_add_sync(0xffffffffu, wn);
    const int base_i = fi - my_i + (int)__reduce_add_sync(0xffffffffu, lane < wid ? wi : 0);
    const int base_n = fn - my_n + (int)__reduce_add_sync(0xffffffffu, lane < wid ? wn : 0);
    // floor(blockIdx.x * tot_i / gridDim.x), and of the next CTA
    const unsigned qi = (unsigned)tot_i / gridDim.x, ri = (unsigned)tot_i % gridDim.x;
    const int i0 = (int)(blockIdx.x * qi + blockIdx.x * ri / gridDim.x);
    const int i1 = (int)((blockIdx.x + 1) * qi + (blockIdx.x + 1) * ri / gridDim.x);
    const bool listing = ulist != nullptr && blockIdx.x == 0 && skip == 0;
    if (listing && tid == 0) *ucount = tot_n;
    // the owners of the range's first and last item say which units (by rank) it spans
    const bool mine = my_i > 0 && base_i < i1 && base_i + my_i > i0;
    auto walk = [&](auto &&f) {
        int i = base_i, r = base_n;
        auto visit = [&](int u, int L, int k) {
            const int n = (k + item_keys - 1) / item_keys;
            if (n == 0) return;
            f(u, L, k, i, n, r);
            i += n;
            ++r;
        };
        if constexpr (HELD > 1) {
#pragma unroll
            for (int j = 0; j < HELD; ++j) visit(u_lo + j, Lh[j], kh[j]);
        } else {
            for (int u = u_lo; u < u_hi; ++u) {
                int L = Lh[0], k = kh[0];
                if (seg > 1) k = keys_of(u, L);
                visit(u, L, k);
            }
        }
    };
    if (mine)
        walk([&](int, int, int, int i, int n, int r) {
            if (i <= i0 && i0 < i + n) pl.first = r;
        });
    __syncthreads();
    const int first = pl.first;
    if (mine || listing)
        walk([&](int u, int L, int k, int i, int n, int r) {
            if (listing) ulist[r] = u;
            const int a = max(i, i0), b = min(i + n, i1);
            if (a >= b) return;
            if (b == i1) pl.n = r - first + 1;
            const int e = r - first - skip;
            if (e < 0 || e >= kPlanRuns) return;
            const int per = item_keys / kTile, t0 = (a - i) * per;
            pl.run[e] = TileRun{u, L, t0, min((b - i) * per, (k + kTile - 1) / kTile) - t0};
        });
    __syncthreads();
    return pl.n;
}

}  // namespace reco
