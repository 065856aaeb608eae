// Bounded search pass, plans whose bounds tie (sm_100a).  The float bounds are computed again for the
// segments that need it (they cost less than storing them would: one addition and one maximum per
// stage), plans within the segment's window are collected per warp, and whenever 32 of them are
// together each lane adds up one walk in the recurrence's own arithmetic (cm_bound.cuh).
// Bound by the chain of a walk's O(S+m) dependent additions wherever plans tie, else by launch and set-up:
// 64 sets of the 64-device job 34 us a phase (most of their layers are equal), 64 of the 256-device job 42
// and 16 us.  Of a CTA's time with ties at 30 stages, the set-up is 11 us, the loop over its segments 1 us
// and one turn of walks, its lanes side by side, 12 us.
//   phase 1: the least of them per segment goes to pick[row]
//   phase 2: those that could still improve on their segment's result go to the list
#include "cm_bound_lane.cuh"

namespace cm {

// What a segment is looked at for.
struct RefineSeg {
    uint64_t lim_bits;   // phase 2: list a plan whose walk costs at most this
    double lim;          // plans whose bound is at most lim ...
    float ev;            //   ... and above ev (what phase 1 has settled already)
    uint32_t scen, tseg, pad;
};
static_assert(sizeof(RefineSeg) <= kRefineSegBytes, "room per segment in bound_dyn_bytes");

// What a segment still needs.  False: nothing.
template <typename T>
__device__ __forceinline__ bool seg_open(const BatchDev &bd, const BoundDev &bo, const BBucket &bk, int phase, uint32_t row, RefineSeg &s) {
    constexpr bool native = std::is_same<T, long long>::value;
    const uint64_t la = bo.lbarg[row], key = bo.pick[row];
    if (la == ~0ull) return false;                                   // nothing fits in memory
    if (key == ~0ull) return false;                                  // part of no strategy within reach
    const float lb = lb_of(la), near = __fmul_ru(lb, 1.0f + kTieWindow);
    const SearchWin w = bo.row_rep ? SearchWin{__uint_as_float((uint32_t)bo.row_lo[row]), 0.0f, ~bo.row_ub[row]} : bo.win[s.scen];
    s.ev = -1.0f;
    s.lim_bits = 0;
    if (phase == 1) {
        s.lim = (double)near;
        return !(lb <= __fmul_rd(w.lo, 1.0f - kTieWindow));          // well below the best step time: any plan will do
    }
    const uint64_t best = bd.seg_best[row];
    if (best == 0) return false;
    const double sb = cost_up(best, native), ub = cost_up(w.ub, native);
    if (sb <= (double)w.lo) return false;
    s.lim = sb < ub ? sb : ub;
    s.lim_bits = best - 1 < w.ub ? best - 1 : w.ub;
    // phase 1 compared everything up to `near` and its choice came out as its walk promised
    if (key < kPickWanted && pick_base(lb, native) + (key >> pick_bits(bk.count)) == best) s.ev = near;
    return (double)lb <= s.lim && s.lim > (double)s.ev;
}

// Lanes 0 .. n-1 take one collected plan each: entry = segment << 8 | thread whose composition it is.
template <typename T>
__device__ __noinline__ void refine_flush(const SProf<T> &sp, const BatchDev &bd, const BoundDev &bo, const BBucket &bk,
                                          int phase, uint64_t tile0, const BoundSmem &sm, const uint32_t *ent, int n) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint32_t e = ent[lane], t = e & 0xffu;
        const SegLite &sg = sm.segs[e >> 8];
        const RefineSeg &rg = reinterpret_cast<const RefineSeg *>(sm.rest)[e >> 8];
        const uint64_t pos = tile0 + (t & (bk.width - 1));
        const CutColumn<kBoundThreads> c{sm.cut - threadIdx.x + t};
        const Walk w = best_walk<T>(sp, c, bk.S, bk.m, sg.tier, sg.n_sync, false);
        const uint64_t bits = Num<T>::bits(walk_cost<T>(sp, c, bk.S, bk.m, sg.tier, sg.n_sync, w));
        if (phase == 1) {
            const float lb = lb_of(bo.lbarg[sg.row]);
            atomicMin(&sm.word[e >> 8], (unsigned long long)pick_key(bits, pick_base(lb, std::is_same<T, long long>::value), pos, pick_bits(bk.count)));
        } else if (bits <= rg.lim_bits) {
            list_append(bd, bo, bk.S <= kRegStagesMax ? 2 : 3, rg.scen, rg.tseg, (uint32_t)pos);
        }
    }
    __syncwarp();
}

template <typename T, int NB, bool UNI_X>
__device__ void refine_body(const SProf<T> &sp, const Tables &tb, const BatchDev &bd, const BoundDev &bo, const BBucket &bk, int phase,
                            uint64_t tile0, int n_act, const BoundSmem &sm, uint32_t *buf /* [64] of this warp */) {
    const int S = bk.S, m = bk.m, W = bk.width;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const int sub = tid / W, n_sub = kBoundThreads / W;
    if (UNI_X) fill_transfers<T, NB>(sm, sp, S, m, n_act);
    const uint64_t pos = tile0 + (tid & (W - 1));
    LaneBound<NB> v;
    v.ok = pos < bk.count;
    if (v.ok) {
        CutWalker w;
        const CutColumn<kBoundThreads> cuts{sm.cut};
        v.ok = make_walker(w, tb, bd.layer_mode, sp.L, S, walk_cand(bd, bk.feas_first, pos), bk.K, tb.mm_slot(S, m)) && cuts.fill(w, S);
        if (v.ok) lane_setup<T, NB, UNI_X>(v, sp, cuts, S, m, bk.feas_first == kNoFeasList, sm.cd);
    }
    __syncthreads();
    const float slack = sp.intval || std::is_same<T, long long>::value ? 1.0f : 0.0f;
    const int n_it = (n_act + n_sub - 1) / n_sub;
    const RefineSeg *rsegs = reinterpret_cast<const RefineSeg *>(sm.rest);
    int n_buf = 0;
    for (int it = 0; it < n_it; ++it) {
        const int s = it * n_sub + sub;
        bool take = false;
        if (s < n_act && v.ok) {
            const float lb = bound_of(lane_value<T, NB, UNI_X>(v, sp, S, m, s, sm), slack);
            take = (double)lb <= rsegs[s].lim && lb > rsegs[s].ev;
        }
        const uint32_t who = __ballot_sync(0xffffffffu, take);
        if (!who) continue;
        if (take) buf[n_buf + __popc(who & ((1u << lane) - 1u))] = ((uint32_t)s << 8) | tid;
        n_buf += __popc(who);
        __syncwarp();
        if (n_buf >= 32) {
            n_buf -= 32;
            refine_flush<T>(sp, bd, bo, bk, phase, tile0, sm, buf + n_buf, 32);
        }
    }
    if (n_buf) refine_flush<T>(sp, bd, bo, bk, phase, tile0, sm, buf, n_buf);
}

template <typename T, bool UNI_X>
__global__ void __launch_bounds__(kBoundThreads) cm_refine_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase) {
    __shared__ SProf<T> sp;
    __shared__ BBucket bks;
    __shared__ uint32_t buf[kBoundThreads / 32][64];
    __shared__ int n_act_s;
    extern __shared__ __align__(16) unsigned char dyn[];
    const uint32_t tid = threadIdx.x;
    if (tid == 0) {
        bks = bo.bucket[bound_bucket(bo, blockIdx.x)];
        n_act_s = lists_full(bd) ? -1 : 0;
    }
    __syncthreads();
    if (n_act_s < 0) return;   // uniform (it only grows from 0)
    const BBucket &bk = bks;
    const BoundJob job = bound_job(bk, blockIdx.x);
    const BoundSmem sm = bound_smem(dyn, bo);
    for (uint32_t q = job.s0 + tid; q < job.s1; q += kBoundThreads) {
        const BoundSeg g = bound_segment(bd, bk, q);
        RefineSeg s;
        s.scen = g.scen; s.tseg = g.tseg; s.pad = 0;
        if (seg_open<T>(bd, bo, bk, phase, g.row, s)) {
            const int at = atomicAdd(&n_act_s, 1);
            sm.segs[at] = seg_lite(tb, g);
            reinterpret_cast<RefineSeg *>(sm.rest)[at] = s;
        }
    }
    __syncthreads();
    const int n_act = n_act_s;
    if (n_act == 0) return;   // uniform
    stage_profile(sp, tb);
    for (int q = tid; q < n_act; q += kBoundThreads) sm.word[q] = ~0ull;
    __syncthreads();
    const int nb = (bk.S + 3) >> 2;
#define CM_NB(K) if (nb <= K) refine_body<T, K, UNI_X>(sp, tb, bd, bo, bk, phase, job.tile0, n_act, sm, buf[tid >> 5]); else
    CM_NB(4) CM_NB(9) CM_NB(16) {}
#undef CM_NB
    if (phase != 1) return;
    __syncthreads();
    for (int q = tid; q < n_act; q += kBoundThreads)
        if (sm.word[q] < bo.pick[sm.segs[q].row]) atomicMin((unsigned long long *)&bo.pick[sm.segs[q].row], sm.word[q]);
}

template <typename T, bool UNI_X>
static cudaError_t launch_refine_one(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(cm_refine_kernel<T, UNI_X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBoundDynMax);
    if (e != cudaSuccess) return e;
    cm_refine_kernel<T, UNI_X><<<bo.n_chunks, kBoundThreads, bo.dyn_bytes, st>>>(t, b, bo, phase);
    return cudaGetLastError();
}
cudaError_t launch_refine(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, cudaStream_t st) {
    if (bo.n_chunks == 0) return cudaSuccess;
    if (native_i64(b)) return bo.uniform_x ? launch_refine_one<long long, true>(t, b, bo, phase, st) : launch_refine_one<long long, false>(t, b, bo, phase, st);
    return bo.uniform_x ? launch_refine_one<double, true>(t, b, bo, phase, st) : launch_refine_one<double, false>(t, b, bo, phase, st);
}

}  // namespace cm
