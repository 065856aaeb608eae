// Bounded search pass, plans whose bounds tie (sm_100a).  The float bounds are computed again for the
// segments that need it (they cost less than storing them would: one addition and one maximum per
// stage), plans within the segment's window are collected per warp, and whenever 32 of them are
// together each lane adds up one walk in the recurrence's own arithmetic (cm_bound.cuh).
//   phase 1: the least of them per segment goes to pick[row]
//   phase 2: those that could still improve on their segment's result go to the list
#include "cm_bound_lane.cuh"

namespace cm {

// What a segment still needs.  False: nothing.
template <typename T>
__device__ __forceinline__ bool seg_open(const BatchDev &bd, const BoundDev &bo, const BBucket &bk, int phase, SegLite &s) {
    constexpr bool native = std::is_same<T, long long>::value;
    const uint64_t la = bo.lbarg[s.row], key = bo.pick[s.row];
    if (la == ~0ull) return false;                                   // nothing fits in memory
    if (bo.window && key == ~0ull) return false;                     // part of no strategy within reach
    const float lb = lb_of(la), near = __fmul_ru(lb, 1.0f + kTieWindow);
    const SearchWin w = bo.window ? bo.win[s.scen] : SearchWin{-1.0f, 0.0f, inf_bits<T>()};
    const bool least = lb <= __fmul_rd(w.lo, 1.0f - kTieWindow);     // well below the best step time: any plan will do
    if (phase == 1) {
        s.lim = (double)near;
        return !least;
    }
    const uint64_t best = bd.seg_best[s.row];
    if (best == 0) return false;
    const double sb = cost_up(best, native), ub = cost_up(w.ub, native);
    if (sb <= (double)w.lo) return false;
    s.lim = sb < ub ? sb : ub;
    s.lim_bits = best - 1 < w.ub ? best - 1 : w.ub;
    // phase 1 compared everything up to `near` and its choice came out as its walk promised
    if (key < kPickWanted && pick_base(lb, native) + (key >> pick_bits(bk.count)) == best) s.ev = near;
    return (double)lb <= s.lim && s.lim > (double)s.ev;
}

struct RefineShared {
    uint64_t a[kBoundThreads], b[kBoundThreads];       // layer composition of every thread (CutEdges)
    uint8_t minmax[kBoundThreads];
    uint32_t buf[kBoundThreads / 32][64];              // per warp: (segment << 8 | thread) of collected plans
};

// Lanes 0 .. n-1 take one collected plan each.
template <typename T>
__device__ __noinline__ void refine_flush(const SProf<T> &sp, const Tables &tb, const BatchDev &bd, const BoundDev &bo, const BBucket &bk,
                                          int phase, uint64_t tile0, const SegLite *segs, unsigned long long *seg_key,
                                          const RefineShared &rs, const uint32_t *ent, int n) {
    const int lane = threadIdx.x & 31;
    if (lane < n) {
        const uint32_t e = ent[lane], t = e & 0xffu;
        const SegLite &sg = segs[e >> 8];
        const uint64_t pos = tile0 + (t & (bk.width - 1));
        CutEdges c{rs.a[t], rs.b[t], nullptr, bd.layer_mode == CM_LAYERS_REMAINDER ? 0 : 1, sp.L / bk.S, sp.L, bk.S};
        if (rs.minmax[t]) { c.kind = 2; c.row = tb.mm_cuts + (size_t)tb.mm_slot(bk.S, bk.m) * (kMaxS + 1); }
        const Walk w = best_walk<T>(sp, c, bk.S, bk.m, sg.tier, sg.n_sync, false);
        const uint64_t bits = Num<T>::bits(walk_cost<T>(sp, c, bk.S, bk.m, sg.tier, sg.n_sync, w));
        if (phase == 1) {
            const float lb = lb_of(bo.lbarg[sg.row]);
            atomicMin(&seg_key[e >> 8], (unsigned long long)pick_key(bits, pick_base(lb, std::is_same<T, long long>::value), pos, pick_bits(bk.count)));
        } else if (bits <= sg.lim_bits) {
            list_append(bd, bo, bk.S <= kRegStagesMax ? 2 : 3, sg.scen, sg.tseg, (uint32_t)pos);
        }
    }
    __syncwarp();
}

template <typename T, int NB, bool UNI_X>
__device__ void refine_body(const SProf<T> &sp, const Tables &tb, const BatchDev &bd, const BoundDev &bo, const BBucket &bk, int phase,
                            uint64_t tile0, const SegLite *segs, int n_act, unsigned long long *seg_key, unsigned char *dyn, RefineShared &rs) {
    const int S = bk.S, m = bk.m, W = bk.width;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const int sub = tid / W, n_sub = kBoundThreads / W;
    float *xs = reinterpret_cast<float *>(dyn);                                            // as in cm_bound.cu
    float *cc = reinterpret_cast<float *>(dyn + bo.dyn_cols) + tid;
    float *dd = cc + S * kBoundThreads;
    uint8_t *cutc = dyn + bo.dyn_cols + sizeof(float) * 2 * S * kBoundThreads + tid;
    const float x1 = __double2float_rd((double)sp.XT[1][0]);
    if (UNI_X) fill_transfers<T, NB>(xs, sp, S, segs, n_act);
    const uint64_t pos = tile0 + (tid & (W - 1));
    LaneBound<NB> v;
    v.ok = pos < bk.count;
    if (v.ok) {
        CutWalker w;
        const uint64_t kappa = walk_kappa(bd.feas, bk.feas_first, pos);
        v.ok = make_walker(w, tb, bd.layer_mode, sp.L, S, kappa, bk.K, tb.mm_slot(S, m));
        rs.a[tid] = w.a; rs.b[tid] = w.b; rs.minmax[tid] = kappa >= bk.K ? 1 : 0;
        if (v.ok) lane_setup<T, NB, UNI_X>(v, sp, cut_edges(w), S, m, bk.feas_first == kNoFeasList, cc, dd, cutc);
    }
    __syncthreads();
    const float slack = sp.intval || std::is_same<T, long long>::value ? 1.0f : 0.0f;
    const int n_it = (n_act + n_sub - 1) / n_sub;
    uint32_t *buf = rs.buf[tid >> 5];
    int n_buf = 0;
    for (int it = 0; it < n_it; ++it) {
        const int s = it * n_sub + sub;
        bool take = false;
        if (s < n_act && v.ok) {
            const SegLite &sg = segs[s];
            const float lb = lane_value<T, NB, UNI_X>(v, sp, S, m, sg, xs + s * 4 * NB, x1, slack, cc, dd, cutc);
            take = (double)lb <= sg.lim && lb > sg.ev;
        }
        const uint32_t who = __ballot_sync(0xffffffffu, take);
        if (!who) continue;
        if (take) buf[n_buf + __popc(who & ((1u << lane) - 1u))] = ((uint32_t)s << 8) | tid;
        n_buf += __popc(who);
        __syncwarp();
        if (n_buf >= 32) {
            n_buf -= 32;
            refine_flush<T>(sp, tb, bd, bo, bk, phase, tile0, segs, seg_key, rs, buf + n_buf, 32);
        }
    }
    if (n_buf) refine_flush<T>(sp, tb, bd, bo, bk, phase, tile0, segs, seg_key, rs, buf, n_buf);
}

template <typename T, bool UNI_X>
__global__ void __launch_bounds__(kBoundThreads) cm_refine_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase) {
    __shared__ SProf<T> sp;
    __shared__ BBucket bks;
    __shared__ RefineShared rs;
    __shared__ int n_act_s;
    extern __shared__ __align__(16) unsigned char dyn[];
    const uint32_t tid = threadIdx.x;
    if (tid == 0) {
        bks = bo.bucket[bound_bucket(bo, blockIdx.x)];
        n_act_s = 0;
    }
    __syncthreads();
    const BBucket &bk = bks;
    const BoundJob job = bound_job(bk, blockIdx.x);
    SegLite *segs = reinterpret_cast<SegLite *>(dyn + bo.dyn_segs);
    unsigned long long *seg_key = reinterpret_cast<unsigned long long *>(dyn + bo.dyn_segs + sizeof(SegLite) * bo.max_group);
    for (uint32_t q = job.s0 + tid; q < job.s1; q += kBoundThreads) {
        SegLite s = seg_lite(tb, bound_segment(bd, bk, q));
        if (seg_open<T>(bd, bo, bk, phase, s)) segs[atomicAdd(&n_act_s, 1)] = s;
    }
    __syncthreads();
    const int n_act = n_act_s;
    if (n_act == 0) return;   // uniform
    stage_profile(sp, tb);
    for (int q = tid; q < n_act; q += kBoundThreads) seg_key[q] = ~0ull;
    __syncthreads();
    const int nb = (bk.S + 3) >> 2;
#define CM_NB(K) if (nb <= K) refine_body<T, K, UNI_X>(sp, tb, bd, bo, bk, phase, job.tile0, segs, n_act, seg_key, dyn, rs); else
    CM_NB(4) CM_NB(9) CM_NB(16) {}
#undef CM_NB
    if (phase != 1) return;
    __syncthreads();
    for (int q = tid; q < n_act; q += kBoundThreads)
        if (seg_key[q] < bo.pick[segs[q].row]) atomicMin((unsigned long long *)&bo.pick[segs[q].row], seg_key[q]);
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
