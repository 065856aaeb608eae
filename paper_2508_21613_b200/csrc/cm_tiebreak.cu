// Tie-break pass of the plan search (sm_100a): among optimal plans the lexicographically smallest
// tuple wins, so each pipeline of a winning (strategy, split) takes the LOWEST layer composition
// that is feasible with cost <= T* (not its own argmin).
#include <algorithm>

#include "cm_bound.cuh"
#include "cm_launch.cuh"
#include "cm_tie_rest.cuh"

namespace cm {

// Rounds of recurrences without success after which a CTA leaves its pipeline to cm_tie_rest_kernel: bounds
// that decide leave one or two candidates, and where they do not (transfers about as long as the stages) tens
// of thousands are left, and a warp each, a few at a time, is the slowest way through them.
constexpr int kTieRoundsWide = 2, kTieRoundsWarp = 6;

// ----------------------------------------------------------------------------------
// A CTA per (winner record, pipeline) walks the segment's candidates upwards, a thread per
// composition: a lower bound above T* rules one out (first in O(stages), then, for those that tie,
// bit for bit along the walk: cm_bound.cuh), and the few that are left are walked by a warp each in
// lock step, lowest first, n_eval of them at a time.  The bound is tight, so about one recurrence
// per pipeline remains; what bounds the kernel is the latency of those, 2(S+m) dependent
// slots.  grid.y: tiles of a segment side by side where the winners alone leave the GPU empty (the
// uncapped spaces hold 10^8 compositions per pipeline); a tile whose first composition is above one
// already found stops.
// ----------------------------------------------------------------------------------
template <typename T, int kTieThreads>
__global__ void __launch_bounds__(kTieThreads) cm_tiebreak_kernel(Tables tb, BatchDev bd, int n_eval) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[kTieThreads / 32][kMaxS + 8];
    __shared__ uint8_t cut_col[kMaxS * kTieThreads];
    __shared__ uint32_t left[kTieThreads / 32];
    __shared__ unsigned long long found;
    const uint32_t b = blockIdx.x / bd.dp_max, p = blockIdx.x % bd.dp_max;
    if (kTieThreads > 32) stage_profile(sp, tb);
    after_previous();
    const Winner &w = bd.winner[b];
    const uint64_t w_bits = w.cost_bits;
    if (w_bits >= inf_bits<T>() || p >= w.dp || lists_full(bd)) return;   // uniform over the CTA
    const SegView g = seg_view(bd, w.scen, w.seg[p]);
    if (g.K == 0) return;                                           // one candidate: known already
    if (kTieThreads <= 32) stage_profile(sp, tb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double goal = std::is_same<T, long long>::value ? __ll2double_ru((long long)w_bits)
                                                          : __longlong_as_double((long long)w_bits);
    unsigned long long *slot = reinterpret_cast<unsigned long long *>(&bd.kappa_sel[(size_t)b * kMaxP + p]);
    const uint64_t count = walk_count(g);
    unsigned long long evaluated = 0;
    int rounds = kTieThreads > 32 ? kTieRoundsWide : kTieRoundsWarp;
    for (uint64_t base = (uint64_t)blockIdx.y * kTieThreads; rounds && base < count; base += (uint64_t)gridDim.y * kTieThreads) {
        __syncthreads();
        if (threadIdx.x == 0) found = *(volatile unsigned long long *)slot;
        __syncthreads();
        if (found <= walk_kappa(bd.feas, g.feas_first, base)) break;   // uniform: this tile and all later ones are higher
        const uint64_t pos = base + threadIdx.x;
        bool maybe = false;
        if (pos < count) {
            CutWalker cw;
            if (make_walker(cw, tb, bd.layer_mode, sp.L, g.S, walk_cand(bd, g.feas_first, pos), g.K, tb.mm_slot(g.S, g.m))) {
                const CutColumn<kTieThreads> c{cut_col + threadIdx.x};
                c.fill(cw, g.S);
                const Walk walk = best_walk<T>(sp, c, g.S, g.m, g.tier, g.n_sync, g.feas_first == kNoFeasList);
                maybe = walk.value >= 0.0 && walk.value <= goal;
                if (maybe && !walk_surely_within(walk.value, goal)) maybe = Num<T>::bits(walk_cost<T>(sp, c, g.S, g.m, g.tier, g.n_sync, walk)) <= w_bits;
            }
        }
        const uint32_t vote = __ballot_sync(0xffffffffu, maybe);
        if (lane == 0) left[warp] = vote;
        __syncthreads();
        if (threadIdx.x == 0) found = ~0ull;
        for (;;) {
            // this warp's candidate: number `warp` among those left, if it is one of the next n_eval
            int skip = warp, at = -1, total = 0;
            for (int q = 0; q < kTieThreads / 32; ++q) {
                const uint32_t v = left[q];
                const int c = __popc(v);
                if (at < 0 && skip < c) at = q * 32 + (int)__fns(v, 0, skip + 1);
                skip -= c;
                total += c;
            }
            __syncthreads();                                        // everybody has read `left`; `found` is reset
            if (total == 0) break;                                  // uniform
            if (warp < n_eval && at >= 0) {
                const Cand cand = walk_cand(bd, g.feas_first, base + at);
                T cost;
                if (warp_plan_cost<T>(sp, tb, bd.layer_mode, g, cand, cuts_s[warp], cost) && lane == 0 &&
                    Num<T>::bits(cost) <= w_bits)
                    atomicMin(&found, (unsigned long long)cand.kappa);
                if (lane == 0) ++evaluated;
            }
            if (threadIdx.x == 0)                                   // strike the candidates being tried
                for (int q = 0, n = n_eval; q < kTieThreads / 32 && n > 0; ++q)
                    while (left[q] && n > 0) { left[q] &= left[q] - 1; --n; }
            __syncthreads();
            if (found != ~0ull || --rounds == 0) break;             // uniform
        }
        if (found != ~0ull) {                                       // the lowest of this tile: later tiles are higher
            if (threadIdx.x == 0) atomicMin(slot, found);
            break;
        }
    }
    if (lane == 0 && evaluated) atomicAdd(&bd.counters[1], evaluated);
    if (threadIdx.x == 0 && rounds == 0 && found == ~0ull && !((atomicOr(&bd.winner[b].open, 1u << p) >> p) & 1u))
        bd.open[atomicAdd(bd.n_open, 1ull) + 1ull] = b * kMaxP + p;   // (the count starts at -1)
}

// ----------------------------------------------------------------------------------
// The same for a batch of shallow pipelines under 1F1B, eight to a warp: the bounds of 32 candidates of one pipeline
// after the other, then the lowest candidate that each has left, all of them at a time in lock step, four lanes each
// (group_plan_cost), until every pipeline has its composition.  A warp of its own keeps six lanes of 32 busy with a pipeline
// of twelve stages: 2576 sets of the 32-device job 57 us, 106 with the kernel above.  Deeper pipelines stay with that
// one: three to a warp wait for the one that needs most attempts (1024 sets of the 256-device job 240 us, 160 above).
// ----------------------------------------------------------------------------------
constexpr int kTieWarps = 2, kTieMost = 8;
// Pipelines from which they share: below, the GPU has room for a warp each, and eight in sequence are the longer chain.
// Batches of the 32-device job, shared and a warp each: 60 sets (300 pipelines) 41 and 18 us, 400 sets 43 and 20, 700 sets 45
// and 33, 1200 sets (6000) 49 and 47, 2500 sets 57 and 90; of the 8-device job, 700 sets (4900) 27 and 23, 1200 sets 29 and 31.
constexpr uint64_t kTieBatchMin = 148 * 44;
constexpr uint32_t kTieTiles = 64;   // of kTile candidates

template <typename T>
__global__ void __launch_bounds__(kTieWarps * 32) cm_tie_batch_kernel(Tables tb, BatchDev bd, uint32_t n_items) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[kTieWarps][kTieMost][kRegStagesMax + 8];   // (per pipeline; none is deeper: launch_tiebreak)
    __shared__ uint8_t cut_col[kTieWarps][kRegStagesMax * 32];
    stage_profile(sp, tb);
    after_previous();
    if (lists_full(bd)) return;   // uniform: no kernel that may run beside this one writes the flag
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int width = 32 / kTieMost;
    const int grp = lane / width, gl = lane - grp * width;
    const uint32_t item0 = (blockIdx.x * kTieWarps + warp) * kTieMost, item = item0 + grp;
    if (item0 >= n_items) return;   // warp-uniform from here on
    // the lane's own pipeline
    bool open = item < n_items;
    const uint32_t b = open ? item / bd.dp_max : 0, p = open ? item % bd.dp_max : 0;
    const Winner &w = bd.winner[b];
    const uint64_t w_bits = w.cost_bits;
    open = open && w_bits < inf_bits<T>() && p < w.dp;
    SegView g{};
    if (open) g = seg_view(bd, w.scen, w.seg[p]);
    open = open && g.K != 0;            // (one candidate: known already)
    const uint32_t count = open ? (uint32_t)walk_count(g) : 0u;   // (launch_tiebreak: few)
    uint32_t base = 0, tile = 0, left = 0, evaluated = 0;
    int rounds = kTieRoundsWarp;
    for (;;) {
        // candidates that its bound does not rule out, for the pipelines that have none left
        uint32_t want;
        while ((want = __ballot_sync(0xffffffffu, open && left == 0)) != 0) {
            const int k = (__ffs((int)want) - 1) / width, from = k * width;
            SegView q;
            q.tier = __shfl_sync(0xffffffffu, g.tier, from);
            q.K = __shfl_sync(0xffffffffu, g.K, from);
            q.feas_first = __shfl_sync(0xffffffffu, g.feas_first, from);
            q.S = __shfl_sync(0xffffffffu, g.S, from);
            q.m = __shfl_sync(0xffffffffu, g.m, from);
            q.n_sync = __shfl_sync(0xffffffffu, g.n_sync, from);
            const uint64_t most = __shfl_sync(0xffffffffu, w_bits, from);
            const uint32_t n = __shfl_sync(0xffffffffu, count, from), first = __shfl_sync(0xffffffffu, base, from);
            const double goal = std::is_same<T, long long>::value ? __ll2double_ru((long long)most) : __longlong_as_double((long long)most);
            bool maybe = false;
            CutWalker cw;
            if (first + lane < n && make_walker(cw, tb, bd.layer_mode, sp.L, q.S, walk_cand(bd, q.feas_first, first + lane), q.K, tb.mm_slot(q.S, q.m))) {
                const CutColumn<32> c{cut_col[warp] + lane};
                c.fill(cw, q.S);
                const Walk walk = best_walk<T>(sp, c, q.S, q.m, q.tier, q.n_sync, q.feas_first == kNoFeasList);
                maybe = walk.value >= 0.0 && walk.value <= goal;
                if (maybe && !walk_surely_within(walk.value, goal))
                    maybe = Num<T>::bits(walk_cost<T>(sp, c, q.S, q.m, q.tier, q.n_sync, walk)) <= most;
            }
            const uint32_t vote = __ballot_sync(0xffffffffu, maybe);
            if (grp == k) {
                left = vote;
                tile = base;
                base += 32;
                if (left == 0 && base >= count) open = false;   // (no candidate within the winning cost: not so for a winner)
            }
        }
        if (!__any_sync(0xffffffffu, open)) break;
        const uint32_t pos = tile + (open ? __ffs((int)left) - 1 : 0);
        left &= left - 1;
        Cand cand{0, 0, 0, false};
        if (open) cand = walk_cand(bd, g.feas_first, pos);
        T cost;
        const bool ok = group_plan_cost<T>(sp, tb, bd.layer_mode, g, cand, open, gl, width, cuts_s[warp][grp], cost);
        const uint32_t hits = __ballot_sync(0xffffffffu, ok && gl == 0 && Num<T>::bits(cost) <= w_bits);
        if (open) {
            if (gl == 0) ++evaluated;
            if ((hits >> (lane - gl)) & 1u) {
                if (gl == 0) bd.kappa_sel[(size_t)b * kMaxP + p] = cand.kappa;   // (the lowest: this warp alone looks, upwards)
                open = false;
            } else if (--rounds == 0) {
                if (gl == 0 && !((atomicOr(&bd.winner[b].open, 1u << p) >> p) & 1u))
                    bd.open[atomicAdd(bd.n_open, 1ull) + 1ull] = b * kMaxP + p;   // (the count starts at -1)
                open = false;
            }
            if (!open) left = 0;
            else if (left == 0 && base >= count) open = false;
        }
    }
    for (int o = 16; o > 0; o >>= 1) evaluated += __shfl_xor_sync(0xffffffffu, evaluated, o);
    if (lane == 0 && evaluated) atomicAdd(&bd.counters[1], (unsigned long long)evaluated);
}

// ----------------------------------------------------------------------------------
// The pipelines that the kernel above has left open, from their lowest candidate on (cm_tie_rest.cuh).  Up to
// kRegStagesMax stages a thread per candidate, its state in registers; 17 .. 48 stages the same with
// a launch per depth (cm_cost_impl.cuh), for which the host has to know that there are any.  Deeper ones, and
// a shortlist's, whose completion the host does not wait for, as above: bounds first and a warp for
// each that is left, but without waiting for one another.
// Bound by issue, as the search pass.  60 sets of a 40-device job, transfers three times the stages (620 000
// candidates, nearly all of 19 and 20 stages): 0.85 ms by depth, 4.5 ms with a warp each, 9 ms if a
// pipeline's tiles stay with four CTAs.  600 sets of the 32-device job over links of 1 GB/s: 9.1 ms a call with
// the kernel above alone, 3.7 with this one.
// ----------------------------------------------------------------------------------
// CTAs: two and four per SM, rounded down to primes.
constexpr int kRestShallow = 293, kRestWarps = 587;

template <typename T>
__global__ void __launch_bounds__(kRestThreads) cm_tie_rest_kernel(Tables tb, BatchDev bd) {
    __shared__ SProf<T> sp;
    const uint32_t n = rest_open(bd);
    if (n == 0) return;
    stage_profile(sp, tb);
    unsigned long long evaluated = 0;
    rest_tiles(bd, n, [](int S) { return S <= kRegStagesMax; }, [&](const RestTile &t) {
        const uint64_t pos = t.base + threadIdx.x;
        unsigned long long hit = ~0ull;
        if (pos < t.count) {
            const Cand cand = walk_cand(bd, t.g.feas_first, pos);
            T cost;
            if (plan_cost_regs_any<T, true>(sp, tb, bd.layer_mode, t.g, cand, cost) && Num<T>::bits(cost) <= t.w_bits) hit = cand.kappa;
            ++evaluated;
        }
        hit = warp_min_u64(hit);
        if ((threadIdx.x & 31) == 0 && hit != ~0ull) t.commit(hit);
    });
    rest_count(bd, evaluated);
}

template <typename T>
__global__ void __launch_bounds__(kRestThreads) cm_tie_rest_warp_kernel(Tables tb, BatchDev bd, int least_stages) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[kRestThreads / 32][kMaxS + 8];
    __shared__ uint8_t cut_col[kMaxS * kRestThreads];
    __shared__ uint32_t left[kRestThreads / 32];
    const uint32_t n = rest_open(bd);
    if (n == 0) return;
    stage_profile(sp, tb);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long evaluated = 0;
    rest_tiles(bd, n, [&](int S) { return S >= least_stages; }, [&](const RestTile &t) {
        const SegView &g = t.g;
        const double goal = std::is_same<T, long long>::value ? __ll2double_ru((long long)t.w_bits) : __longlong_as_double((long long)t.w_bits);
        const uint64_t pos = t.base + threadIdx.x;
        bool maybe = false;
        CutWalker cw;
        if (pos < t.count && make_walker(cw, tb, bd.layer_mode, sp.L, g.S, walk_cand(bd, g.feas_first, pos), g.K, tb.mm_slot(g.S, g.m))) {
            const CutColumn<kRestThreads> c{cut_col + threadIdx.x};
            c.fill(cw, g.S);
            const Walk walk = best_walk<T>(sp, c, g.S, g.m, g.tier, g.n_sync, g.feas_first == kNoFeasList);
            maybe = walk.value >= 0.0 && walk.value <= goal;
            if (maybe && !walk_surely_within(walk.value, goal)) maybe = Num<T>::bits(walk_cost<T>(sp, c, g.S, g.m, g.tier, g.n_sync, walk)) <= t.w_bits;
        }
        const uint32_t vote = __ballot_sync(0xffffffffu, maybe);
        if (lane == 0) left[warp] = vote;
        __syncthreads();
        // this warp's: every fourth of those left, upwards
        bool more = true;
        for (int q = 0, k = 0; q < kRestThreads / 32 && more; ++q)
            for (uint32_t v = left[q]; v && more; v &= v - 1, ++k) {
                if (k % (kRestThreads / 32) != warp) continue;
                const Cand cand = walk_cand(bd, g.feas_first, t.base + q * 32 + __ffs((int)v) - 1);
                const unsigned long long so_far = __shfl_sync(0xffffffffu, (unsigned long long)*t.slot, 0);
                if (so_far <= cand.kappa) { more = false; continue; }
                T cost;
                if (warp_plan_cost<T>(sp, tb, bd.layer_mode, g, cand, cuts_s[warp], cost) && lane == 0 && Num<T>::bits(cost) <= t.w_bits)
                    t.commit(cand.kappa);
                if (lane == 0) ++evaluated;
                __syncwarp();
            }
    });
    rest_count(bd, evaluated);
}

cudaError_t launch_tie_rest(const Tables &t, const BatchDev &b, uint64_t stages, bool by_depth, cudaStream_t st, int *launches) {
    if (b.B <= 0 || b.max_tiles_per_seg == 0 || b.dp_max == 0) return cudaSuccess;
    const bool native = native_i64(b);
    if (stages & ((1ull << kRegStagesMax) - 1ull)) {
        if (native) cm_tie_rest_kernel<long long><<<kRestShallow, kRestThreads, 0, st>>>(t, b);
        else cm_tie_rest_kernel<double><<<kRestShallow, kRestThreads, 0, st>>>(t, b);
        ++*launches;
    }
    for (int S = kRegStagesMax + 1; by_depth && S <= kWideStagesMax; ++S)
        if ((stages >> (S - 1)) & 1ull) {
            const cudaError_t e = launch_tie_rest_deep(t, b, S, st);
            if (e != cudaSuccess) return e;
            ++*launches;
        }
    const int least = by_depth ? kWideStagesMax + 1 : kRegStagesMax + 1;
    if (stages >> (least - 1)) {
        if (native) cm_tie_rest_warp_kernel<long long><<<kRestWarps, kRestThreads, 0, st>>>(t, b, least);
        else cm_tie_rest_warp_kernel<double><<<kRestWarps, kRestThreads, 0, st>>>(t, b, least);
        ++*launches;
    }
    return cudaGetLastError();
}

cudaError_t launch_tiebreak(const Tables &t, const BatchDev &b, uint64_t stages, cudaStream_t st) {
    if (b.B <= 0 || b.max_tiles_per_seg == 0 || b.dp_max == 0) return cudaSuccess;
    const uint64_t nx = (uint64_t)b.B * b.dp_max;
    if (nx >= (1ull << 31)) return cudaErrorInvalidConfiguration;
    // A failure handled on its own: a wide CTA per pipeline, whose warps try candidates side by side.  A
    // batch: a warp per pipeline; the first 32 compositions nearly always hold the answer, and the first
    // that its bound leaves nearly always is it.  1024 sets of the 256-device job: 133 us with a warp, 172 us with
    // two, where a plan-per-lane kernel per depth took 1300 us in all.
    const bool wide = nx <= 148 * 2;
    // Several pipelines to a warp where there are many, of few tiles each (a long walk would hold up the others).
    if (nx >= kTieBatchMin && t.sched != CM_SCHED_GPIPE && b.max_tiles_per_seg <= kTieTiles && !(stages >> kRegStagesMax)) {
        const unsigned ctas = (unsigned)((nx + kTieMost * kTieWarps - 1) / (kTieMost * kTieWarps));
        return native_i64(b) ? launch_next(cm_tie_batch_kernel<long long>, ctas, kTieWarps * 32, 0, st, t, b, (uint32_t)nx)
                             : launch_next(cm_tie_batch_kernel<double>, ctas, kTieWarps * 32, 0, st, t, b, (uint32_t)nx);
    }
    const unsigned threads = wide ? 256 : 32;
    const int n_eval = wide ? 256 / 32 : 1;
    const uint64_t tiles = ((uint64_t)b.max_tiles_per_seg * kTile + threads - 1) / threads;
    uint64_t y = (148 * 4 + nx - 1) / nx;
    y = std::min<uint64_t>(std::min(y, tiles), 65535);
    const dim3 grid((unsigned)nx, (unsigned)std::max<uint64_t>(y, 1), 1);
    if (native_i64(b))
        return wide ? launch_next(cm_tiebreak_kernel<long long, 256>, grid, threads, 0, st, t, b, n_eval)
                    : launch_next(cm_tiebreak_kernel<long long, 32>, grid, threads, 0, st, t, b, n_eval);
    return wide ? launch_next(cm_tiebreak_kernel<double, 256>, grid, threads, 0, st, t, b, n_eval)
                : launch_next(cm_tiebreak_kernel<double, 32>, grid, threads, 0, st, t, b, n_eval);
}

}  // namespace cm
