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

// Runs skip .. skip + kPlanRuns of this CTA's range into pl.run; returns the range's runs.
// Given ulist, CTA 0 also lists every unit with work (ascending) and their count; given err_len, it
// reports lengths out of range, also of units that the mask leaves out.  All threads of the CTA call
// it; it starts and ends with a CTA barrier.
__device__ __forceinline__ int plan_runs(TilePlan &pl, const int32_t *__restrict__ lens, const ScoreMask &mask, int w,
                                         int L_cap, int units, bool candidates_only, int item_keys, int skip,
                                         int32_t *ulist, int32_t *ucount, unsigned *err_len)
{
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
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
    int my_i = 0, my_n = 0;
#pragma unroll 4
    for (int u = u_lo; u < u_hi; ++u) {
        int L;
        const int k = keys_of(u, L);
        my_i += (k + item_keys - 1) / item_keys;
        my_n += k > 0;
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
    int base_i = fi - my_i, base_n = fn - my_n, tot_i = 0, tot_n = 0;
    for (int k = 0; k < nw; ++k) {
        if (k < wid) {
            base_i += pl.items[k];
            base_n += pl.units[k];
        }
        tot_i += pl.items[k];
        tot_n += pl.units[k];
    }
    const int i0 = (int)((long long)blockIdx.x * tot_i / gridDim.x);
    const int i1 = (int)((long long)(blockIdx.x + 1) * tot_i / gridDim.x);
    const bool listing = ulist != nullptr && blockIdx.x == 0 && skip == 0;
    if (listing && tid == 0) *ucount = tot_n;
    // the owners of the range's first and last item say which units (by rank) it spans
    const bool mine = my_i > 0 && base_i < i1 && base_i + my_i > i0;
    auto walk = [&](auto &&f) {
        int i = base_i, r = base_n;
        for (int u = u_lo; u < u_hi; ++u) {
            int L;
            const int k = keys_of(u, L), n = (k + item_keys - 1) / item_keys;
            if (n == 0) continue;
            f(u, L, k, i, n, r);
            i += n;
            ++r;
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
