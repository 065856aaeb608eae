// Micro-batch splits of a strategy under the remainder rule, a warp per strategy.  The rule hands one more
// micro-batch to R of the pipelines, every choice of them a split, so the least step time of a strategy
// follows from the two costs of each pipeline without going through its splits: the least value t among
// them such that the pipelines that cannot do with their smaller share (cost above t) number at most R,
// those that can take the larger one (cost at most t) number at least R, and the former are among the
// latter; C(may - must, R - must) splits then stay within t.
#pragma once

#include "cm_device.cuh"

namespace cm {

// Row of a pipeline's segment, the first occurrence of pipelines that strategies have in common.
__device__ __forceinline__ uint32_t canon_row(const BatchDev &bd, const Tmpl &tp, const Scen &sc, const Strat &s, int p, int k) {
    uint32_t t = s.seg_first + p * s.n_m + k;
    if (bd.tseg_canon) t = bd.tseg_canon[t];
    return sc.seg_base + (t - tp.tseg_first);
}

// The two costs of every pipeline of a strategy, a lane each: lane 2p + k holds pipeline p with its
// smaller (k = 0) or larger share (2 kMaxP = 32 lanes).  get(row): the cost of a segment's row.
template <typename Get>
__device__ __forceinline__ uint64_t strat_cost(const BatchDev &bd, const Tmpl &tp, const Scen &sc, const Strat &s, uint64_t inf, Get get) {
    const int p = (threadIdx.x & 31) >> 1, k = threadIdx.x & 1;
    uint64_t v = inf;
    if (p < s.dp && k < s.n_m && s.m_lo[p] + k >= 1) v = get(canon_row(bd, tp, sc, s, p, k));
    return v < inf ? v : inf;
}

// Is there a split of the strategy within this lane's t, and how many?
__device__ __forceinline__ bool splits_within(uint64_t v, int dp, int R, uint64_t t, int &free_ones, int &left) {
    int may = 0, must = 0;
    bool ok = true;
    for (int p = 0; p < dp; ++p) {
        const bool need = __shfl_sync(0xffffffffu, v, 2 * p) > t, can = __shfl_sync(0xffffffffu, v, 2 * p + 1) <= t;
        may += can;
        must += need;
        ok = ok && (can || !need);
    }
    free_ones = may - must;
    left = R - must;
    return ok && left >= 0 && may >= R;
}

// Least step time above `after` (~0: any) of a strategy, in every lane.
__device__ __forceinline__ uint64_t strat_best(uint64_t v, const Strat &s, uint64_t after, uint64_t inf) {
    const int lane = threadIdx.x & 31, dp = s.dp, R = s.R;
    const bool mine = lane < 2 * dp;
    if (after == ~0ull) {
        // Where no pipeline is cheaper with the larger share (always so for bounds, and for results that
        // are all there): everybody's smaller share, and the R cheapest larger ones.
        const uint64_t other = __shfl_xor_sync(0xffffffffu, v, 1);
        if (!R || __all_sync(0xffffffffu, !mine || (lane & 1 ? v >= other : v <= other))) {
            uint64_t t = ~warp_min_u64(mine && !(lane & 1) ? ~v : ~0ull);   // largest of the smaller shares
            if (R) {
                int below = 0;
                for (int p = 0; p < dp; ++p) {
                    const uint64_t h = __shfl_sync(0xffffffffu, v, 2 * p + 1);
                    below += h < v || (h == v && 2 * p + 1 < lane);
                }
                const uint32_t who = __ballot_sync(0xffffffffu, mine && (lane & 1) && below == R - 1);
                const uint64_t at = who ? __shfl_sync(0xffffffffu, v, __ffs(who) - 1) : inf;
                t = at > t ? at : t;
            }
            return t;
        }
    }
    int f, l;
    const bool ok = splits_within(v, dp, R, v, f, l) && mine && v < inf && (after == ~0ull || v > after);
    return warp_min_u64(ok ? v : inf);
}

// The same in 32 bits (bounds, 0xffffffff: none), for N strategies at a time: three dependent loads each, all of them
// in flight together.  row_of(row): the row that is searched for a row.
template <int N, typename RowOf>
__device__ __forceinline__ void strat_bounds(const BatchDev &bd, const Tmpl &tp, const Scen &sc, const Strat *strat, uint32_t first, uint32_t step,
                                             const uint64_t *lbarg, RowOf row_of, uint32_t (&v)[N]) {
    const int p = (threadIdx.x & 31) >> 1, k = threadIdx.x & 1;
    uint32_t t[N];
    bool ok[N];
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const uint32_t si = first + u * step;
        const Strat &s = strat[si < tp.n_strat ? si : 0];
        ok[u] = si < tp.n_strat && p < s.dp && k < s.n_m && s.m_lo[p] + k >= 1;
        t[u] = ok[u] ? s.seg_first + p * s.n_m + k : tp.tseg_first;
    }
    if (bd.tseg_canon) {
#pragma unroll
        for (int u = 0; u < N; ++u) t[u] = bd.tseg_canon[t[u]];
    }
#pragma unroll
    for (int u = 0; u < N; ++u) t[u] = row_of(sc.seg_base + (t[u] - tp.tseg_first));
#pragma unroll
    for (int u = 0; u < N; ++u) {
        const uint32_t w = (uint32_t)(lbarg[t[u]] >> 32);
        v[u] = ok[u] ? w : 0xffffffffu;
    }
}
// Least step time of a strategy from its bounds: strat_best, whose first case they nearly always are.
__device__ __forceinline__ uint32_t strat_best_bound(uint32_t v, const Strat &s) {
    const int lane = threadIdx.x & 31, dp = s.dp, R = s.R;
    const bool mine = lane < 2 * dp;
    const uint32_t other = __shfl_xor_sync(0xffffffffu, v, 1);
    if (R && !__all_sync(0xffffffffu, !mine || (lane & 1 ? v >= other : v <= other))) return (uint32_t)strat_best(v, s, ~0ull, 0xffffffffull);
    uint32_t t = __reduce_max_sync(0xffffffffu, mine && !(lane & 1) ? v : 0u);   // largest of the smaller shares
    if (R) {
        int below = 0;
        for (int p = 0; p < dp; ++p) {
            const uint32_t h = __shfl_sync(0xffffffffu, v, 2 * p + 1);
            below += h < v || (h == v && 2 * p + 1 < lane);
        }
        const uint32_t who = __ballot_sync(0xffffffffu, mine && (lane & 1) && below == R - 1);
        const uint32_t at = who ? __shfl_sync(0xffffffffu, v, __ffs((int)who) - 1) : 0xffffffffu;
        t = at > t ? at : t;
    }
    return t;
}

}  // namespace cm
