// Bounded search pass, plans whose bounds tie (sm_100a).  The float bounds are computed again for the
// segments that need it (they cost less than storing them would: one addition and one maximum per
// dear boundary), plans within the segment's window are collected per CTA, and its threads add up one walk
// each in the recurrence's own arithmetic (cm_bound.cuh).
// Bound by the chain of a walk's O(S+m) dependent additions wherever plans tie, else by launch and set-up:
// 64 sets of the 64-device job 30 and 25 us (most of their layers are equal), 1024 of the 256-device job 37 and 31,
// 2576 of the 32-device job 30 and 29.  Of a CTA's time with ties at 30 stages, the set-up is 11 us, the loop over its
// segments 1 us and one turn of walks, its threads side by side, 12 us.
//   phase 1: the least of them per segment goes to pick[row]
//   phase 2: those that could still improve on their segment's result go to the list
#include <algorithm>

#include "cm_bound_lane.cuh"

namespace cm {

// What a segment is looked at for.
struct RefineSeg {
    uint64_t lim_bits;   // phase 2: list a plan whose walk costs at most this
    float lim;           // plans whose bound is at most lim ...
    float ev;            //   ... and above ev (what phase 1 has settled already)
    uint32_t scen, tseg;
    int n_sync;
};
// What a segment still needs; least: the least bound among the compositions at hand, or one below it.  False: nothing.
template <typename T>
__device__ __forceinline__ bool seg_open(const BatchDev &bd, const BoundDev &bo, const BBucket &bk, int phase, uint32_t row, float least, RefineSeg &s) {
    constexpr bool native = std::is_same<T, long long>::value;
    const uint64_t la = bo.lbarg[row], key = bo.pick[row];
    if (la == ~0ull) return false;                                   // nothing fits in memory
    if (key == ~0ull) return false;                                  // part of no strategy within reach
    const float lb = lb_of(la), near = __fmul_ru(lb, 1.0f + kTieWindow);
    const SearchWin w = bo.row_rep ? SearchWin{__uint_as_float((uint32_t)bo.row_lo[row]), 0.0f, ~bo.row_ub[row]} : bo.win[s.scen];
    s.ev = -1.0f;
    s.lim_bits = 0;
    if (phase == 1) {
        s.lim = near;
        return least <= near && !(lb <= __fmul_rd(w.lo, 1.0f - kTieWindow));          // well below the best step time: any plan will do
    }
    const uint64_t best = bd.seg_best[row];
    if (best == 0) return false;
    const double sb = cost_up(best, native), ub = cost_up(w.ub, native);
    if (sb <= (double)w.lo) return false;
    s.lim = __double2float_rd(sb < ub ? sb : ub);   // (bounds are floats: none lies between)
    s.lim_bits = best - 1 < w.ub ? best - 1 : w.ub;
    // phase 1 compared everything up to `near` and its choice came out as its walk promised
    if (key < kPickWanted && pick_base(lb, native) + (key >> pick_bits(bk.count)) == best) s.ev = near;
    return least <= s.lim && s.lim > s.ev;
}

// Segments that are gone through at a time, and, where parts with open segments are listed, the size of a part: plans tie by
// the hundred in some parts while most are empty, so small parts spread them over the CTAs.
constexpr int kRefineSegs = 32;
static_assert(kBoundThreads == 128, "queue entries");

// Shared memory of a CTA: the segments that are open, and the cuts of its compositions.
struct RefineSmem {
    SegLite segs[kBoundSegs];
    SegHot hot[kBoundSegs];
    RefineSeg open[kBoundSegs];
    unsigned long long word[kBoundSegs];   // phase 1: least walk cost
    int n_queue;
    bool full;                             // the lists, when the segments were looked at
    uint16_t queue[kRefineSegs * kBoundThreads];   // plans to walk: segment << 7 | thread whose composition it is
};

// A plan's walk, added up in the recurrence's own arithmetic: segment s, composition of thread c.
template <typename T>
__device__ __noinline__ void refine_walk(const SProf<T> &sp, const BatchDev &bd, const BoundDev &bo, const BBucket &bk,
                                         int phase, uint64_t tile0, RefineSmem &sm, uint8_t *cuts, int s, int c) {
    const SegLite &sg = sm.segs[s];
    const RefineSeg &rg = sm.open[s];
    const uint64_t pos = tile0 + c;
    const CutColumn<kBoundThreads> cc{cuts + c};
    const Walk w = best_walk<T>(sp, cc, bk.S, bk.m, sg.tier, rg.n_sync, false);
    const uint64_t bits = Num<T>::bits(walk_cost<T>(sp, cc, bk.S, bk.m, sg.tier, rg.n_sync, w));
    if (phase == 1) {
        const float lb = lb_of(bo.lbarg[sg.row]);
        atomicMin(&sm.word[s], (unsigned long long)pick_key(bits, pick_base(lb, std::is_same<T, long long>::value), pos, pick_bits(bk.count)));
    } else if (bits <= rg.lim_bits) {
        list_append(bd, bo, bk.S <= kRegStagesMax ? 2 : 3, rg.scen, rg.tseg, (uint32_t)pos);
    }
}

// A part of the segments that CTA `cta` of cm_bound_kernel took, `size` of them.
struct RefineJob : BoundJob { uint32_t base; };
__device__ __forceinline__ RefineJob refine_job(const BBucket &bk, uint32_t cta, uint32_t part, uint32_t size) {
    RefineJob j;
    static_cast<BoundJob &>(j) = bound_job(bk, cta);
    j.base = j.s0 + part * size;
    j.s1 = min(j.s1, j.base + size);
    return j;
}
template <typename T>
__device__ __forceinline__ bool thread_open(const BatchDev &bd, const BoundDev &bo, const BBucket &bk, const RefineJob &job, int phase, SegRec &g, RefineSeg &s) {
    const uint32_t q = job.base + threadIdx.x;
    if (q >= job.s1) return false;
    const float least = bo.tile_min ? bo.tile_min[bk.min_first + job.tile * bk.n_seg + q] : 0.0f;
    g = bo.rec[bk.seg_first + q];
    s.scen = g.scen; s.tseg = g.tseg; s.n_sync = g.n_sync;
    return seg_open<T>(bd, bo, bk, phase, g.row, least, s);
}

// The parts that have open segments, listed: most have none, and a CTA of the kernel below takes a quarter of an SM
// whether it has or not (1024 sets of the 256-device job, phase 2: 64 us for its 7368 CTAs, most of them empty).
template <typename T>
__global__ void __launch_bounds__(kBoundThreads) cm_open_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase) {
    __shared__ BBucket bks;
    const uint32_t cta = blockIdx.x / bo.parts, part = blockIdx.x - cta * bo.parts;
    find_bucket(bo, cta, &bks);
    __syncthreads();
    after_previous();
    if (lists_full(bd)) return;   // uniform: no kernel that may run beside this one writes the flag
    SegRec g;
    RefineSeg s;
    const bool open = thread_open<T>(bd, bo, bks, refine_job(bks, cta, part, kBoundSegs), phase, g, s);
    if (__any_sync(0xffffffffu, open) && (threadIdx.x & 31) == 0)   // (a warp's segments are a part; counts start at -1)
        bo.work[atomicAdd(&bo.count[3 + phase], 1u) + 1u] = blockIdx.x * (kBoundSegs / kRefineSegs) + (threadIdx.x >> 5);
}

// Few segments are open: here the lanes keep a composition each.
// ahead: the composition while the kernel before this one ends (phase 1 only).
// Whether the lists are full is ONE thread's look, which the CTA acts on together: in phase 2 the CTAs of this
// very kernel set the flag, and warps that each looked for themselves could part ways at the barriers below.  (In phase
// 1 nothing has been listed yet.)
template <typename T, bool UNI_X>
__device__ __forceinline__ void refine_part(const Tables &tb, const BatchDev &bd, const BoundDev &bo, int phase, uint32_t item, uint32_t size, bool ahead,
                                            SProf<T> &sp, BBucket &bks, RefineSmem &sm, int &n_open, unsigned char *dyn) {
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const uint32_t per_cta = bo.parts * (kBoundSegs / size), cta = item / per_cta, part = item - cta * per_cta;
    find_bucket(bo, cta, &bks);
    if (ahead) stage_profile(sp, tb);
    if (tid == 0) n_open = 0;
    __syncthreads();
    const BBucket &bk = bks;
    const RefineJob job = refine_job(bk, cta, part, size);
    if (!ahead) after_previous();
    const int S = bk.S, W = bk.width, dear = dear_tier(tb);
    unsigned char *term_col = dyn + tid * kTermSize<UNI_X>;
    uint8_t *cuts = dyn + bo.dyn_cuts;
    const bool any = (int)tid < W && job.tile0 + tid < bk.count;
    Cand cand{0, 0, 0, false};
    if (any) cand = walk_cand(bd, bk.feas_first, job.tile0 + tid);   // (on its way while the segments are looked at)
    LaneBound v;
    if (ahead) {
        v = lane_of<T, UNI_X, true>(sp, tb, bd, bk, any, cand, dear, term_col, cuts + tid);
        after_previous();
    }
    const bool full = tid == 0 && phase == 2 && lists_full(bd);   // (on its way with the segments)
    SegRec g;
    RefineSeg rs;
    if (thread_open<T>(bd, bo, bk, job, phase, g, rs)) {
        const int at = atomicAdd(&n_open, 1);
        sm.segs[at] = seg_lite(g.tier, g.row, g.n_sync, tb.prof->bw_sync);
        sm.open[at] = rs;
        sm.word[at] = ~0ull;
    }
    if (tid == 0) sm.full = full;
    __syncthreads();
    const int n_act = n_open;
    if (n_act == 0 || sm.full) return;   // uniform
    if (!ahead) {
        stage_profile(sp, tb);
        __syncthreads();
        v = lane_of<T, UNI_X, true>(sp, tb, bd, bk, any, cand, dear, term_col, cuts + tid);
    }
    const float delta = dear_extra(sp, dear), slack = sp.intval || std::is_same<T, long long>::value ? 1.0f : 0.0f;
    if ((int)tid < n_act) sm.hot[tid] = seg_hot<UNI_X>(sm.segs[tid], S, dear, delta, sp.sched == CM_SCHED_GPIPE);
    // plans within their segment's limits are collected, then walked, a thread each
    for (int s0 = 0; s0 < n_act; s0 += kRefineSegs) {
        __syncthreads();   // (the segments' data; nobody reads an earlier queue any more)
        if (tid == 0) sm.n_queue = 0;
        __syncthreads();
        for (int s = s0; s < n_act && s < s0 + kRefineSegs; ++s) {
            bool take = false;
            if (v.ok) {
                const float lb = bound_of(bound_value_of<UNI_X>(v, term_col, sm.hot[s], delta), slack);
                take = lb <= sm.open[s].lim && lb > sm.open[s].ev;
            }
            const uint32_t who = __ballot_sync(0xffffffffu, take);
            if (!who) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(&sm.n_queue, __popc(who));
            at = __shfl_sync(0xffffffffu, at, 0) + __popc(who & ((1u << lane) - 1u));
            if (take) sm.queue[at] = (uint16_t)(((s - s0) << 7) | tid);
        }
        __syncthreads();
        for (int k = tid; k < sm.n_queue; k += kBoundThreads)
            refine_walk<T>(sp, bd, bo, bk, phase, job.tile0, sm, cuts, s0 + (sm.queue[k] >> 7), sm.queue[k] & 127);
    }
    if (phase != 1) return;
    __syncthreads();
    if ((int)tid < n_act && sm.word[tid] < bo.pick[sm.segs[tid].row]) atomicMin((unsigned long long *)&bo.pick[sm.segs[tid].row], sm.word[tid]);
}

template <typename T, bool UNI_X>
__global__ void __launch_bounds__(kBoundThreads) cm_refine_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase) {
    __shared__ SProf<T> sp;
    __shared__ BBucket bks;
    __shared__ RefineSmem sm;
    __shared__ int n_open;
    extern __shared__ __align__(16) unsigned char dyn[];
    if (bo.few) {
        // (there is nearly always something to compare in phase 1, and nearly never in phase 2)
        refine_part<T, UNI_X>(tb, bd, bo, phase, blockIdx.x, kBoundSegs, phase == 1, sp, bks, sm, n_open, dyn);
        return;
    }
    after_previous();
    if (!bo.work) {
        refine_part<T, UNI_X>(tb, bd, bo, phase, blockIdx.x, kBoundSegs, false, sp, bks, sm, n_open, dyn);
        return;
    }
    const uint32_t n = bo.count[3 + phase] + 1u;
    for (uint32_t k = blockIdx.x; k < n; k += gridDim.x) {
        refine_part<T, UNI_X>(tb, bd, bo, phase, bo.work[k], kRefineSegs, false, sp, bks, sm, n_open, dyn);
        __syncthreads();
    }
}

template <typename T, bool UNI_X>
static cudaError_t launch_refine_one(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, cudaStream_t st, int *launches) {
    cudaError_t e = cudaFuncSetAttribute(cm_refine_kernel<T, UNI_X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBoundDynMax);
    if (e != cudaSuccess) return e;
    const unsigned items = bo.n_chunks * bo.parts;
    const bool listed = !bo.few && bo.work;
    if (listed) {
        e = launch_next(cm_open_kernel<T>, items, kBoundThreads, 0, st, t, b, bo, phase);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    ++*launches;
    return launch_next(cm_refine_kernel<T, UNI_X>, listed ? std::min(items, 148u * 4) : items, kBoundThreads, bo.dyn_refine, st, t, b, bo, phase);
}
cudaError_t launch_refine(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, cudaStream_t st, int *launches) {
    if (bo.n_chunks == 0) return cudaSuccess;
    if (native_i64(b)) return bo.uniform_x ? launch_refine_one<long long, true>(t, b, bo, phase, st, launches) : launch_refine_one<long long, false>(t, b, bo, phase, st, launches);
    return bo.uniform_x ? launch_refine_one<double, true>(t, b, bo, phase, st, launches) : launch_refine_one<double, false>(t, b, bo, phase, st, launches);
}

}  // namespace cm
