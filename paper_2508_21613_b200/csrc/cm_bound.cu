// Bounded search pass (sm_100a): least cost per segment without running the recurrence on every
// pipeline-plan.
//
//   cm_bound_kernel    lower bound of every plan of every segment, the least one per segment
//   cm_window_kernel   per scenario: the step times that can still be the answer, and the segments of
//                      the strategies that can reach them
//   cm_refine_kernel   compares plans whose bounds tie, bit for bit (cm_refine.cu; cm_open_kernel lists the
//                      parts of a large layout that have any)
//   cm_gather_kernel   lists the most promising plan of every segment needed
//   cm_list_*_kernel   the recurrence on the listed plans
//
// The sequence is: bounds -> window from the bounds -> refine (phase 1) -> gather -> recurrence ->
// window from the results -> refine (phase 2) -> recurrence.  Phase 1 is optimistic: it assumes that a
// bound is met by its plan, as it nearly always is, and takes ONE plan per segment: the one of least
// bound, near-ties told apart by the exact sum along their walks.  Phase 2 is the proof: every plan
// that its bound does not exclude is listed, which is normally none.
//
// Why a plan may stay out, with T* the scenario's best step time and lo <= T* <= ub:
//   - its segment belongs to no strategy whose step time from bounds alone is at most ub;
//   - its bound is above ub: its segment cannot be part of the answer through it;
//   - its segment has a plan with a result of at most lo: the slowest pipeline decides a step time, so
//     for every (strategy, split) that includes the segment a smaller minimum changes nothing;
//   - its bound is not below its segment's result so far.
// Every per-segment minimum of a strategy that can win is then exact, or at most lo, or (rightly)
// above ub, and the split reduction returns the same winner as with all minima exact.  For a shortlist
// of k pairs, ub is the k-th best step time.  A segment that scenarios share goes by the least lo and the
// largest ub of the scenarios it is marked for (1000 sets of the 256-device job, searched with sharing:
// 1190 us when this came, 963 now; with the segment's own result for ub and nothing for lo 2380 us, or, where
// bounds miss and the lists overflow, 8200 us).
#include <algorithm>

#include "cm_bound_lane.cuh"
#include "cm_split.cuh"

namespace cm {

// Bound by look-ups in shared memory and by set-up: 1024 sets of the 256-device job (75 million plans) 140 us, 795
// with a term per stage and a reduction over lanes per segment (201 thread-instructions a plan), 270 with a term per
// dear boundary and the lanes still a composition each; 2576 sets of the 32-device job (24 million) 56 us, 210 before.
// A CTA holds the terms of up to kBoundThreads compositions (a thread sets up one) and takes its group of segments
// by them, kBoundSegs at a time, a lane per segment: the lane has the places of its segment's dear boundaries in
// registers and goes through the compositions, one look-up, addition and maximum per dear boundary and no
// reduction over lanes.  The warps share the compositions (or, where these are few, the segments).
template <bool UNI_X, int NF>
__device__ __forceinline__ unsigned long long least_bound(const float4 *comp, const unsigned char *terms, const SegHot &h, float delta, int c0, int c1) {
    float least = __uint_as_float(0x7f800000u);
    int at = 0;
#pragma unroll 4
    for (int c = c0; c < c1; ++c) {
        const float4 v = comp[c];
        const float value = bound_value<UNI_X, NF>(v.x, v.y, v.z, terms + c * kTermSize<UNI_X>, h, delta);
        if (value < least) { least = value; at = c; }
    }
    return ((unsigned long long)__float_as_uint(least) << 32) | (uint32_t)at;
}

// Segments up to which, where one of them crosses more dear boundaries than are kept in a list, the lanes keep a composition
// each and go through the segments, with a reduction per segment: a lane per segment leaves most lanes idle there and goes
// through 32 compositions in a long chain (one failure of the 64-device job, a device per node and up to 47 dear
// boundaries: 198 us a call with a lane per segment, 161 up to 8 segments, 149 up to 32).  A short chain takes the same either
// way (256-device job, 4 dear boundaries: 139 and 139, 12 sets of it 268 with a lane per segment, 275 up to 32).
constexpr int kFewSegs = 32;
template <bool UNI_X>   // (out of line: the kernel's other path is the one that most calls take)
__device__ __noinline__ void least_of_lanes(const LaneBound &v, const unsigned char *term_col, const SegHot *segs, int n_seg, float delta, unsigned long long *word) {
    const uint32_t lane = threadIdx.x & 31;
    for (int s = 0; s < n_seg; ++s) {
        const uint32_t value = __float_as_uint(bound_value_of<UNI_X>(v, term_col, segs[s], delta));
        const uint32_t least = __reduce_min_sync(0xffffffffu, value), who = __ballot_sync(0xffffffffu, value == least);
        if (lane == 0) word[s] = ((unsigned long long)least << 32) | (threadIdx.x + __ffs((int)who) - 1);
    }
}

template <typename T, bool UNI_X>
__global__ void __launch_bounds__(kBoundThreads) cm_bound_kernel(Tables tb, BatchDev bd, BoundDev bo) {
    __shared__ SProf<T> sp;
    __shared__ BBucket bks;
    __shared__ float4 comp[kBoundThreads];
    __shared__ SegLite segs[kBoundSegs];
    __shared__ unsigned long long word[kBoundThreads / 32][kBoundSegs];
    __shared__ SegHot few[kFewSegs];
    __shared__ bool long_chain;   // a segment crosses more dear boundaries than a list holds (looked at where it matters)
    extern __shared__ __align__(16) unsigned char terms[];
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    find_bucket(bo, blockIdx.x, &bks);
    stage_profile(sp, tb);
    if (tid == 0) long_chain = false;
    __syncthreads();
    const BBucket &bk = bks;
    const BoundJob job = bound_job(bk, blockIdx.x);
    const int S = bk.S, m = bk.m, W = bk.width, dear = dear_tier(tb);
    const uint32_t tile0 = (uint32_t)job.tile0;   // (positions are 32-bit)
    const bool any = (int)tid < W && tile0 + tid < bk.count;
    Cand cand{0, 0, 0, false};
    if (any) cand = walk_cand(bd, bk.feas_first, tile0 + tid);   // (on its way while the segments are looked up)
    auto take_segments = [&](uint32_t base, int n_seg) {
        if ((int)tid >= n_seg) return;
        const BoundSeg g = bound_segment(bd, bk, base + tid);
        segs[tid] = seg_lite(g.tier, g.row, g.n_sync, sp.bw_sync);
        if (n_seg <= kFewSegs && __popcll(dear_bits(g.tier, dear, S)) > kDearMax) long_chain = true;   // (nothing else is written)
        if (job.tile == 0) bo.rec[bk.seg_first + base + tid] = seg_record(g);
    };
    LaneBound v;
    if (bo.few) {   // the compositions while the kernel before this one ends
        v = lane_of<T, UNI_X, false>(sp, tb, bd, bk, any, cand, dear, terms + tid * kTermSize<UNI_X>, nullptr);
        after_previous();
    } else {
        after_previous();
    }
    take_segments(job.s0, (int)min(job.s1 - job.s0, (uint32_t)kBoundSegs));
    if (!bo.few) v = lane_of<T, UNI_X, false>(sp, tb, bd, bk, any, cand, dear, terms + tid * kTermSize<UNI_X>, nullptr);
    comp[tid] = make_float4(v.best, v.u0, v.g, 0.0f);
    const float delta = dear_extra(sp, dear), slack = sp.intval || std::is_same<T, long long>::value ? 1.0f : 0.0f;
    const bool gpipe = sp.sched == CM_SCHED_GPIPE;
    const int n_ok = __syncthreads_count(v.ok);
    if (tid == 0 && n_ok) {   // what this pass decides: the plans, and the cells recurrences over them would take
        const unsigned long long plans = (unsigned long long)n_ok * (unsigned long long)(job.s1 - job.s0);
        const unsigned long long cells = bk.role == 2 ? 0ull
            : bk.role == 1 ? 2ull * S * (m + 1) + 3ull * S * (S - 1) / 2 : 2ull * S * m;
        atomicAdd(&bd.counters[0], plans * cells);
        atomicAdd(&bd.counters[2], plans);
    }
    const int parts = W > 64 ? 4 : W > 32 ? 2 : 1, part = warp % parts;   // of the compositions
    const int c0 = part * 32, c1 = W < 32 ? W : c0 + 32;
    for (uint32_t base = job.s0; base < job.s1; base += kBoundSegs) {
        const int n_seg = (int)min(job.s1 - base, (uint32_t)kBoundSegs);
        if (base > job.s0) {
            take_segments(base, n_seg);
            __syncthreads();
        }
        const bool comp_lanes = n_seg <= kFewSegs && long_chain;   // uniform
        if (comp_lanes) {
            if ((int)tid < n_seg) few[tid] = seg_hot<UNI_X>(segs[tid], S, dear, delta, gpipe);
            __syncthreads();
            if ((int)warp < parts) least_of_lanes<UNI_X>(v, terms + tid * kTermSize<UNI_X>, few, n_seg, delta, word[warp]);
        }
        for (int g = warp / parts * 32; g < n_seg && !comp_lanes; g += 128 / parts) {
            const SegHot h = seg_hot<UNI_X>(segs[min(g + (int)lane, n_seg - 1)], S, dear, delta, gpipe);
            unsigned long long key;
#define CM_NF(N) case N: key = least_bound<UNI_X, N>(comp, terms, h, delta, c0, c1); break;
            switch (__reduce_max_sync(0xffffffffu, h.n)) {
                CM_NF(0) CM_NF(1) CM_NF(2) CM_NF(3) CM_NF(4) CM_NF(5) CM_NF(6)
            default: key = least_bound<UNI_X, -1>(comp, terms, h, delta, c0, c1);
            }
#undef CM_NF
            word[part][g + lane] = key;
        }
        __syncthreads();
        if ((int)tid < n_seg) {
            unsigned long long least = word[0][tid];
            for (int w = 1; w < parts; ++w) least = word[w][tid] < least ? word[w][tid] : least;
            const float value = __uint_as_float((uint32_t)(least >> 32)), lb = bound_of(value, slack);
            if (bo.tile_min) bo.tile_min[bk.min_first + job.tile * bk.n_seg + base + tid] = lb;
            if (value < __uint_as_float(0x7f800000u)) {
                least = ((unsigned long long)__float_as_uint(lb) << 32) | (tile0 + (uint32_t)least);
                unsigned long long *row = (unsigned long long *)&bo.lbarg[segs[tid].row];
                if (least < *row) atomicMin(row, least);
            }
        }
        __syncthreads();
    }
}
static_assert(kDearMax == 6, "the cases above");

// Segments that a CTA takes by one set of compositions: setting those up costs about as much as 128 segments.
constexpr int kBoundGroup = 384;
int bound_group() { return kBoundGroup; }
// Dynamic shared memory: terms; cm_refine_kernel, from dyn_cuts on, cuts [stages][threads] bytes.
size_t bound_dyn_bytes(BoundDev &bo, int max_stages, bool uniform_x) {
    const size_t terms = (size_t)max_stages * kTermRow * (uniform_x ? kTermSize<true> : kTermSize<false>);
    bo.dyn_cuts = (uint32_t)terms;
    bo.dyn_bytes = terms;
    bo.dyn_refine = terms + (size_t)max_stages * kBoundThreads;
    return bo.dyn_refine;
}

template <typename T, bool UNI_X>
static cudaError_t launch_bound_one(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(cm_bound_kernel<T, UNI_X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBoundDynMax);
    if (e != cudaSuccess) return e;
    return launch_next(cm_bound_kernel<T, UNI_X>, bo.n_chunks, kBoundThreads, bo.dyn_bytes, st, t, b, bo);
}
cudaError_t launch_bound(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    if (bo.n_chunks == 0) return cudaSuccess;
    if (native_i64(b)) return bo.uniform_x ? launch_bound_one<long long, true>(t, b, bo, st) : launch_bound_one<long long, false>(t, b, bo, st);
    return bo.uniform_x ? launch_bound_one<double, true>(t, b, bo, st) : launch_bound_one<double, false>(t, b, bo, st);
}

// ----------------------------------------------------------------------------------
// Window of a scenario: the best step time of any of its strategies (cm_split.cuh), from the bounds
// (phase 0) or the results (phase 1).  Either then marks the segments of the strategies whose step time
// from bounds is still within reach.
// ----------------------------------------------------------------------------------
// Phase 0 marks strategies this far above the best step time from bounds: one plan of each of their
// segments is evaluated, so that a result that misses its bound a little still leaves phase 2 nothing to do.
constexpr float kReach = 1.0f / (1 << 13);

__device__ __forceinline__ uint64_t block_min_u64(uint64_t v /* warp-uniform */, uint64_t *red) {
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) v = red[w] < v ? red[w] : v;
    return v;
}

// Strategies whose step times from bounds are kept from the first look to the second.
constexpr uint32_t kWinKept = 2048;

__global__ void __launch_bounds__(1024) cm_window_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase, int k_best, uint64_t inf_cost) {
    __shared__ uint64_t red[32];
    __shared__ unsigned long long total;
    __shared__ uint32_t kept[kWinKept];
    __shared__ uint32_t n_listed;
    __shared__ SearchWin was;
    const uint32_t b = blockIdx.x;
    const Scen sc = bd.scen[b];
    const Tmpl tp = bd.tmpl[sc.tmpl];
    const Strat *strat = bd.strat + tp.strat_first;
    const uint32_t warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31;
    after_previous();
    const uint64_t inf = phase ? inf_cost : 0xffffffffull;
    if (threadIdx.x == 0) {
        n_listed = 0;
        if (phase) was = bo.win[b];
    }
    __syncthreads();
    // From results, only the strategies that the bounds had within reach can have any step time below infinity
    // that counts: their segments are the ones that were evaluated.
    const bool by_list = phase && was.n_strat <= (uint32_t)kWinStrats;
    const uint32_t n_look = by_list ? was.n_strat : tp.n_strat;
    auto look_at = [&](uint32_t q) -> const Strat & { return strat[by_list ? was.strat[q] : q]; };
    auto row_of = [&](uint32_t own) { return bo.row_rep ? bo.row_rep[own] : own; };
    auto cost_of = [&](const Strat &s, int from_results, uint64_t most) {
        return strat_cost(bd, tp, sc, s, most, [&](uint32_t own) {
            const uint32_t row = row_of(own);
            return from_results ? bd.seg_best[row] : (uint64_t)(bo.lbarg[row] >> 32);
        });
    };
    constexpr int kSide = 4;   // strategies side by side in a warp
    uint64_t first = ~0ull, t = ~0ull;
    bool enough = false;
    for (int r = 0; r < k_best && !enough; ++r) {
        uint64_t mine = inf;
        if (!phase && r == 0) {
            uint32_t v[kSide], least = 0xffffffffu;
            for (uint32_t si = warp; si < tp.n_strat; si += kSide * warps) {
                strat_bounds<kSide>(bd, tp, sc, strat, si, warps, bo.lbarg, row_of, v);
#pragma unroll
                for (int u = 0; u < kSide; ++u) {
                    const uint32_t at = si + u * warps;
                    if (at >= tp.n_strat) break;   // uniform
                    const uint32_t best = strat_best_bound(v[u], strat[at]);
                    if (lane == 0 && at < kWinKept) kept[at] = best;
                    least = best < least ? best : least;
                }
            }
            mine = least;
        } else {
            for (uint32_t q = warp; q < n_look; q += warps) {
                const Strat &s = look_at(q);
                const uint64_t v = strat_best(cost_of(s, phase, inf), s, t, inf);
                mine = v < mine ? v : mine;
            }
        }
        t = block_min_u64(mine, red);
        if (r == 0) first = t;
        if (t >= inf || k_best == 1) break;
        if (threadIdx.x == 0) total = 0;
        __syncthreads();
        for (uint32_t q = warp; q < n_look; q += warps) {
            const Strat &s = look_at(q);
            int f, l;
            const bool ok = splits_within(cost_of(s, phase, inf), s.dp, s.R, t, f, l);
            if (ok && lane == 0) atomicAdd(&total, (unsigned long long)binom_at(tb.binom, f, l));
        }
        __syncthreads();
        enough = total >= (unsigned long long)k_best;
        __syncthreads();
    }
    if (k_best > 1 && !enough && t < inf) t = inf;
    float lo = 0.0f;
    float reach = -1.0f;   // step times from bounds up to here (-1: none)
    bool relist = true;    // the strategies within reach are listed
    if (phase) {
        reach = __double2float_ru(cost_up(t, native_i64_dev(bd)));
        lo = was.lo;
        if (threadIdx.x == 0) bo.win[b].ub = t;
        // (uniform) phase 0 has marked them all: the results came out as promised
        if (reach <= was.reach && !bo.row_rep) return;
        relist = !(reach <= was.reach && by_list);
    } else {
        lo = first < inf ? __uint_as_float((uint32_t)first) : 0.0f;
        if (first < inf) reach = t < inf ? __fmul_ru(__uint_as_float((uint32_t)t), 1.0f + kReach) : __uint_as_float(0x7f800000u);
        if (threadIdx.x == 0) { bo.win[b].lo = lo; bo.win[b].reach = reach; bo.win[b].ub = inf_cost; }
    }
    __syncthreads();   // (what was kept)
    auto mark = [&](uint32_t si, uint32_t best) {   // a strategy and its step time from bounds, warp-uniform
        if (best == 0xffffffffu || __uint_as_float(best) > reach) return;
        const Strat &s = strat[si];
        if (relist && lane == 0) {
            const uint32_t at = atomicAdd(&n_listed, 1u);
            if (at < (uint32_t)kWinStrats) bo.win[b].strat[at] = (uint16_t)si;   // (longer lists, and numbers beyond 16 bits, go unused)
        }
        const int p = lane >> 1, k = lane & 1;
        if (p >= s.dp || k >= s.n_m) return;
        const uint32_t row = row_of(canon_row(bd, tp, sc, s, p, k));
        // a bound beyond reach: not part of the answer through this share (where results move the reach up, the
        // second window marks again)
        if (lb_of(bo.lbarg[row]) > reach) return;
        if (bo.row_rep) {
            const unsigned long long l = __float_as_uint(lo), u = ~t;   // (u: of a result, phase 1)
            if (l < bo.row_lo[row]) atomicMin((unsigned long long *)&bo.row_lo[row], l);
            if (phase && u < bo.row_ub[row]) atomicMin((unsigned long long *)&bo.row_ub[row], u);
        }
        if (bo.pick[row] == ~0ull) bo.pick[row] = kPickWanted;   // (every writer writes the same)
    };
    if (!phase && tp.n_strat <= kWinKept) {
        for (uint32_t si = warp; si < tp.n_strat; si += warps) { mark(si, kept[si]); __syncwarp(); }
    } else if (!relist) {
        for (uint32_t q = warp; q < was.n_strat; q += warps) {
            const Strat &s = strat[was.strat[q]];
            mark(was.strat[q], (uint32_t)strat_best(cost_of(s, 0, 0xffffffffull), s, ~0ull, 0xffffffffull));
            __syncwarp();
        }
    } else {
        uint32_t v[kSide];
        for (uint32_t si = warp; si < tp.n_strat; si += kSide * warps) {
            strat_bounds<kSide>(bd, tp, sc, strat, si, warps, bo.lbarg, row_of, v);
#pragma unroll
            for (int u = 0; u < kSide; ++u) {
                const uint32_t at = si + u * warps;
                if (at >= tp.n_strat) break;   // uniform
                mark(at, strat_best_bound(v[u], strat[at]));
                __syncwarp();
            }
        }
    }
    if (!relist) return;
    __syncthreads();
    if (threadIdx.x == 0) bo.win[b].n_strat = n_listed <= (uint32_t)kWinStrats && tp.n_strat <= 0x10000u ? n_listed : kWinAll;
}

cudaError_t launch_window(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, int k_best, cudaStream_t st) {
    if (b.B <= 0) return cudaSuccess;
    // A warp per four strategies, latency of their dependent loads.  Up to a scenario per SM the CTA takes them all at
    // once; beyond, CTAs of an SM stand in for one another (with one strategy at a time: 64 sets of the 64-device job
    // 10 us with 1024 threads, 16 with 256; 515 sets of the 32-device job 28 us with 256 threads, 37 with 1024).
    // Four at a time, kept for the marking and listed for later: 2576 sets of the 32-device job 95 -> 54 us from
    // bounds, 88 -> 52 from results (where most have to be marked again), 515 sets 26 -> 16 and 17 -> 4.
    return launch_next(cm_window_kernel, b.B, b.B <= 148 ? 1024 : 256, 0, st, t, b, bo, phase, k_best, batch_inf_bits(b));
}

// ----------------------------------------------------------------------------------
// The plan that phase 1 takes per segment: a thread per searched segment.
// ----------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) cm_gather_kernel(Tables tb, BatchDev bd, BoundDev bo) {
    const uint32_t at = blockIdx.x * 128 + threadIdx.x;
    after_previous();
    if (at >= bo.n_segs) return;
    const SegRec g = bo.rec[at];
    const uint64_t la = bo.lbarg[g.row], key = bo.pick[g.row];
    if (la == ~0ull || key == ~0ull) return;   // nothing fits in memory / not needed
    const TSeg &ts = bd.tseg[g.tseg];
    const uint64_t count = ts.feas_first != kNoFeasList ? (uint64_t)ts.feas_count : ts.K ? ts.K + 1 : 1;
    const uint32_t pos = key == kPickWanted ? (uint32_t)la : (uint32_t)(key & ((1ull << pick_bits(count)) - 1ull));
    list_append(bd, bo, ts.S <= kRegStagesMax ? 0 : 1, g.scen, g.tseg, pos);
}

cudaError_t launch_gather(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    if (bo.n_segs == 0) return cudaSuccess;
    return launch_next(cm_gather_kernel, (bo.n_segs + 127) / 128, 128, 0, st, t, b, bo);
}

// ----------------------------------------------------------------------------------
// The recurrence on the listed plans.  Pipelines of at most 16 stages: a thread per plan, state in
// registers; deeper ones in lock step, 2(S+m) slots (a thread would need ~100 us for its chain of 2 S m cells): a
// warp per plan up to two and a half plans for each of its 2960 warps, three plans per warp (two beyond 40 stages) beyond:
// few groups of three leave most warps idle (passes of the 256-device job, a plan and three per warp: 140 sets, 3058 plans, 204
// and 244 us, 260 sets, 5625 plans, 286 and 310, 350 sets, 7509 plans, 348 and 349, 1000 sets, 21375 plans, 792 and 759).
// ----------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t list_length(const BoundDev &bo, int list) {
    const uint32_t n = bo.count[list] + 1u, room = bo.list_first[list + 1] - bo.list_first[list];
    return n < room ? n : room;
}
template <typename T> __device__ __forceinline__ void list_commit(const BatchDev &bd, uint32_t row, T cost) {
    const uint64_t bits = Num<T>::bits(cost);
    if (bits < bd.seg_best[row]) atomicMin((unsigned long long *)&bd.seg_best[row], (unsigned long long)bits);
}
// work: cells in the low 40 bits, plans above
__device__ __forceinline__ void count_list_work(const BatchDev &bd, unsigned long long work) {
    for (int o = 16; o > 0; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
    if ((threadIdx.x & 31) == 0 && work) {
        atomicAdd(&bd.counters[3], work & ((1ull << 40) - 1ull));
        atomicAdd(&bd.counters[5], work >> 40);
    }
}

constexpr uint32_t kListAhead = 148;   // CTAs that fetch the profile before they know whether the list is long enough for them
template <typename T>
__global__ void __launch_bounds__(kChunk) cm_list_shallow_kernel(Tables tb, BatchDev bd, BoundDev bo, int list) {
    __shared__ SProf<T> sp;
    if (blockIdx.x < kListAhead) stage_profile(sp, tb);
    after_previous();
    const uint32_t n = list_length(bo, list);
    if ((uint64_t)blockIdx.x * kChunk >= n || lists_full(bd)) return;
    if (blockIdx.x >= kListAhead) stage_profile(sp, tb);
    __syncthreads();
    const uint4 *entries = bo.list + bo.list_first[list];
    unsigned long long work = 0;
    for (uint32_t i = blockIdx.x * kChunk + threadIdx.x; i < n; i += gridDim.x * kChunk) {
        const uint4 e = entries[i];
        const SegView g = seg_view(bd, e.x, e.y);
        const Cand cand = walk_cand(bd, g.feas_first, e.z);
        T cost;
        const bool ok = g.m >= g.S - 1 ? plan_cost_regs_any<T>(sp, tb, bd.layer_mode, g, cand, cost)
                                       : plan_cost_regs_any<T, true>(sp, tb, bd.layer_mode, g, cand, cost);
        if (ok) list_commit<T>(bd, g.row, cost);
        work += 2ull * g.S * g.m + (1ull << 40);
    }
    count_list_work(bd, work);
}

template <typename T>
__global__ void __launch_bounds__(kChunk, 5) cm_list_deep_kernel(Tables tb, BatchDev bd, BoundDev bo, int list) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[kChunk / 32][4][kMaxS + 8];   // (per plan; the fourth: lanes without one)
    if (blockIdx.x < kListAhead) stage_profile(sp, tb);
    after_previous();
    const uint32_t n = list_length(bo, list);
    if ((uint64_t)blockIdx.x * (kChunk / 32) >= n || lists_full(bd)) return;
    if (blockIdx.x >= kListAhead) stage_profile(sp, tb);
    __syncthreads();
    const uint4 *entries = bo.list + bo.list_first[list];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_warps = gridDim.x * (kChunk / 32), first = blockIdx.x * (kChunk / 32) + warp;
    unsigned long long work = 0;
    if (2ull * n <= 5ull * n_warps || sp.sched == CM_SCHED_GPIPE) {
        for (uint32_t i = first; i < n; i += n_warps) {
            const uint4 e = entries[i];
            const SegView g = seg_view(bd, e.x, e.y);
            T cost;
            if (warp_plan_cost<T>(sp, tb, bd.layer_mode, g, walk_cand(bd, g.feas_first, e.z), cuts_s[warp][0], cost) && lane == 0)
                list_commit<T>(bd, g.row, cost);
            if (lane == 0) work += 2ull * g.S * g.m + (1ull << 40);
        }
    } else {
        for (uint32_t i0 = 3 * first; i0 < n; i0 += 3 * n_warps)
            for (uint32_t i = i0; i < i0 + 3 && i < n;) {   // those of equal depth together
                const int S = bd.tseg[entries[i].y].S, width = (S + 3) >> 2, most = 32 / width < 3 ? 32 / width : 3;
                const int grp = lane / width, gl = lane - grp * width;
                const uint32_t at = i + grp;
                const bool here = grp < most && at < i0 + 3 && at < n;
                const uint4 e = entries[here ? at : i];
                const uint32_t other = __ballot_sync(0xffffffffu, !here || bd.tseg[e.y].S != S);
                const int k = other ? (__ffs((int)other) - 1) / width : most;   // (lanes without a plan come last)
                const SegView g = seg_view(bd, entries[grp < k ? at : i].x, entries[grp < k ? at : i].y);
                const uint4 mine = entries[grp < k ? at : i];
                T cost;
                if (group_plan_cost<T>(sp, tb, bd.layer_mode, g, walk_cand(bd, g.feas_first, mine.z), grp < k, gl, width, cuts_s[warp][grp < 3 ? grp : 3], cost) &&
                    gl == 0)
                    list_commit<T>(bd, g.row, cost);
                if (gl == 0 && grp < k) work += 2ull * g.S * g.m + (1ull << 40);
                i += k;
            }
    }
    count_list_work(bd, work);
}

cudaError_t launch_lists(const Tables &t, const BatchDev &b, const BoundDev &bo, int first_list, cudaStream_t st, int *launches) {
    const uint64_t shallow = bo.list_first[first_list + 1] - bo.list_first[first_list];
    const uint64_t deep = bo.list_first[first_list + 2] - bo.list_first[first_list + 1];
    cudaError_t e = cudaSuccess;
    if (shallow) {
        const unsigned grid = (unsigned)std::min<uint64_t>((shallow + kChunk - 1) / kChunk, 148 * 4);
        e = native_i64(b) ? launch_next(cm_list_shallow_kernel<long long>, grid, kChunk, 0, st, t, b, bo, first_list)
                          : launch_next(cm_list_shallow_kernel<double>, grid, kChunk, 0, st, t, b, bo, first_list);
        ++*launches;
    }
    if (deep && e == cudaSuccess) {
        const unsigned grid = (unsigned)std::min<uint64_t>((deep + kChunk / 32 - 1) / (kChunk / 32), 148 * 5);
        e = native_i64(b) ? launch_next(cm_list_deep_kernel<long long>, grid, kChunk, 0, st, t, b, bo, first_list + 1)
                          : launch_next(cm_list_deep_kernel<double>, grid, kChunk, 0, st, t, b, bo, first_list + 1);
        ++*launches;
    }
    return e;
}

}  // namespace cm
