// cm_evaluate (sm_100a): cost and feasibility of single candidates of a space, in whatever order the
// caller lists them.
//
//   shallow spaces (at most 16 stages)   a thread per candidate, everything in registers
//   deep spaces, few candidates          a warp per candidate in lock step
//   deep spaces, many candidates         binned: cm_evaluate_bin_kernel checks the memory of every
//       candidate and lists the feasible ones by depth, then every depth runs the register-resident
//       recurrence of the search (a thread per candidate, stage times in a shared-memory column)
//
// The recurrence needs its state in registers, hence a depth known at compile time; a thread with
// run-time depth keeps it in local memory, at a tenth of the rate (200 000 candidates of the 256-device
// job: 7.57 ms that way, 0.42 ms binned).
#include <algorithm>

#include "cm_eval_out.cuh"

namespace cm {

// Template segment that owns candidate e of the space's one scenario, -1 past the end.
__device__ __forceinline__ int candidate_segment(const BatchDev &bd, const EvalDev &ev, uint64_t e) {
    if (e >= ev.n_cand) return -1;
    const Tmpl tp = bd.tmpl[bd.scen[0].tmpl];
    const TSeg *seg = bd.tseg + tp.tseg_first;
    uint32_t lo = 0, hi = tp.n_tseg - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (seg[mid].cand_first <= e) lo = mid; else hi = mid - 1;
    }
    return (int)(tp.tseg_first + lo);
}
__device__ __forceinline__ uint64_t candidate_at(const EvalDev &ev, uint64_t t) { return ev.idx ? ev.idx[t] : ev.first + t; }

template <typename T>
__global__ void __launch_bounds__(128) cm_evaluate_shallow_kernel(Tables tb, BatchDev bd, EvalDev ev) {
    __shared__ SProf<T> sp;
    stage_profile(sp, tb);
    __syncthreads();
    const uint64_t t = (uint64_t)blockIdx.x * 128 + threadIdx.x;
    if (t >= ev.count) return;
    const uint64_t e = candidate_at(ev, t);
    const int s = candidate_segment(bd, ev, e);
    T c = Num<T>::inf();
    bool ok = false;
    if (s >= 0) {
        const SegView g = seg_view(bd, 0, (uint32_t)s);
        const Cand cand{e - bd.tseg[s].cand_first, 0, 0, false};
        T v;
        ok = g.m >= g.S - 1 ? plan_cost_regs_any<T>(sp, tb, bd.layer_mode, g, cand, v)
                            : plan_cost_regs_any<T, true>(sp, tb, bd.layer_mode, g, cand, v);
        if (ok) c = v;
    }
    eval_out<T>(bd, ev, t, ok, c);
}

template <typename T>
__global__ void __launch_bounds__(128) cm_evaluate_warp_kernel(Tables tb, BatchDev bd, EvalDev ev) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[4][kMaxS + 8];
    stage_profile(sp, tb);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t t = (uint64_t)blockIdx.x * 4 + warp;
    if (t >= ev.count) return;
    const uint64_t e = candidate_at(ev, t);
    const int s = candidate_segment(bd, ev, e);
    T c = Num<T>::inf();
    bool ok = false;
    if (s >= 0) {
        T v;
        ok = warp_plan_cost<T>(sp, tb, bd.layer_mode, seg_view(bd, 0, (uint32_t)s), Cand{e - bd.tseg[s].cand_first, 0, 0, false}, cuts_s[warp], v);
        if (ok) c = v;
    }
    if (lane == 0) eval_out<T>(bd, ev, t, ok, c);
}

// Memory check and binning of one round of candidates.
template <typename T>
__global__ void __launch_bounds__(128) cm_evaluate_bin_kernel(Tables tb, BatchDev bd, EvalDev ev) {
    __shared__ SProf<T> sp;
    stage_profile(sp, tb);
    __syncthreads();
    const uint32_t slot = blockIdx.x * 128 + threadIdx.x;
    const uint64_t t = ev.base + slot;
    const bool have = slot < ev.slab && t < ev.count;
    int region = -1;
    uint4 entry = make_uint4(0, 0, 0, 0);
    if (have) {
        const uint64_t e = candidate_at(ev, t);
        const int s = candidate_segment(bd, ev, e);
        if (s >= 0) {
            const TSeg g = bd.tseg[s];
            const uint64_t kappa = e - g.cand_first;
            CutWalker w;
            bool ok = g.m >= 1 && make_walker(w, tb, bd.layer_mode, sp.L, g.S, Cand{kappa, 0, 0, false}, g.K, tb.mm_slot(g.S, g.m));
            // (the mask of a remainder composition rides along, so that nobody unranks it again)
            const bool masked = ok && w.kind == 0;
            const uint64_t word = masked ? w.a : kappa;
            const uint32_t flags = masked ? kEvalMasked : 0u;
            int lo = 0;
            for (int i = 0; i < g.S && ok; ++i) {
                const int hi = w.next();
                ok = hi > lo && stage_fits(sp.PS[hi] - sp.PS[lo], sp.PA[hi] - sp.PA[lo], i, g.S, g.m, sp.cap, sp.sched);
                lo = hi;
            }
            if (ok) {
                region = g.S <= kRegStagesMax ? kEvalShallow : g.S <= kWideStagesMax ? (int)g.S : kEvalRest;
                entry = make_uint4(slot | flags, (uint32_t)s, (uint32_t)word, (uint32_t)(word >> 32));
            }
        }
        if (region < 0) eval_out<T>(bd, ev, t, false, Num<T>::inf());
    }
    const uint32_t mates = __match_any_sync(0xffffffffu, region), lane = threadIdx.x & 31;
    const int lead = __ffs(mates) - 1;
    uint32_t at = 0;
    if (region >= 0 && (int)lane == lead) at = atomicAdd(&ev.n_list[region], (uint32_t)__popc(mates));
    at = __shfl_sync(0xffffffffu, at, lead) + __popc(mates & ((1u << lane) - 1u));
    if (region >= 0) eval_region(ev, region)[at] = entry;
}

template <typename T>
__global__ void __launch_bounds__(128) cm_evaluate_list_shallow_kernel(Tables tb, BatchDev bd, EvalDev ev) {
    __shared__ SProf<T> sp;
    const uint32_t n = ev.n_list[kEvalShallow];
    if ((uint64_t)blockIdx.x * 128 >= n) return;
    stage_profile(sp, tb);
    __syncthreads();
    for (uint32_t i = blockIdx.x * 128 + threadIdx.x; i < n; i += gridDim.x * 128) {
        const EvalEntry x = eval_entry(bd, ev, kEvalShallow, i);
        T c;
        const bool ok = x.g.m >= x.g.S - 1 ? plan_cost_regs_any<T>(sp, tb, bd.layer_mode, x.g, x.cand, c)
                                           : plan_cost_regs_any<T, true>(sp, tb, bd.layer_mode, x.g, x.cand, c);
        eval_out<T>(bd, ev, x.t, ok, ok ? c : Num<T>::inf());
    }
}

template <typename T>
__global__ void __launch_bounds__(128) cm_evaluate_list_warp_kernel(Tables tb, BatchDev bd, EvalDev ev) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[4][kMaxS + 8];
    const uint32_t n = ev.n_list[kEvalRest];
    if ((uint64_t)blockIdx.x * 4 >= n) return;
    stage_profile(sp, tb);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint32_t i = blockIdx.x * 4 + warp; i < n; i += gridDim.x * 4) {
        const EvalEntry x = eval_entry(bd, ev, kEvalRest, i);
        T c;
        const bool ok = warp_plan_cost<T>(sp, tb, bd.layer_mode, x.g, x.cand, cuts_s[warp], c);
        if (lane == 0) eval_out<T>(bd, ev, x.t, ok, ok ? c : Num<T>::inf());
    }
}

// One-candidate policies: the cost cm_policy_kernel left behind.
__global__ void cm_evaluate_single_kernel(BatchDev bd, EvalDev ev, int policy, uint64_t inf) {
    const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= ev.count) return;
    const uint64_t c = candidate_at(ev, t) == 0 ? bd.pol_cost[policy] : inf;
    eval_out_bits(bd, ev, t, c < inf, c);
}

static int eval_region_list(uint64_t stages, int *out) {   // regions a space needs, deepest first
    int n = 0;
    if (stages >> kWideStagesMax) out[n++] = kEvalRest;
    for (int S = kWideStagesMax; S > kRegStagesMax; --S)
        if ((stages >> (S - 1)) & 1ull) out[n++] = S;
    if (stages & ((1ull << kRegStagesMax) - 1ull)) out[n++] = kEvalShallow;
    return n;
}

uint64_t eval_workspace(uint64_t stages, uint32_t *slab) {
    if (!(stages >> kRegStagesMax)) return 0;
    int regions[kEvalRegions];
    const int n = eval_region_list(stages, regions);
    *slab = std::min(kEvalSlabMax, std::max(kEvalListMax / (uint32_t)n, 1u << 15)) & ~127u;
    return (uint64_t)n * *slab + kEvalRegions;   // (a counter takes an entry: plenty)
}

template <typename T>
static cudaError_t evaluate_binned(const Tables &t, const BatchDev &b, EvalDev ev, uint64_t stages, uint4 *workspace, cudaStream_t st,
                                   const SideStreams *side) {
    int regions[kEvalRegions];
    const int n = eval_region_list(stages, regions);
    eval_workspace(stages, &ev.slab);
    ev.n_list = reinterpret_cast<uint32_t *>(workspace);
    ev.list = workspace + kEvalRegions;
    for (int q = 0; q < n; ++q) ev.place[regions[q]] = (uint8_t)q;
    const int n_side = side ? std::min(side->n, n - 1) : 0;
    for (ev.base = 0; ev.base < ev.count; ev.base += ev.slab) {
        const uint64_t round = std::min<uint64_t>(ev.slab, ev.count - ev.base);
        cudaError_t e = cudaMemsetAsync(ev.n_list, 0, kEvalRegions * sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
        cm_evaluate_bin_kernel<T><<<(unsigned)((round + 127) / 128), 128, 0, st>>>(t, b, ev);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        if (n_side > 0) {
            e = cudaEventRecord(side->fork, st);
            for (int k = 0; k < n_side && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(side->stream[k], side->fork, 0);
            if (e != cudaSuccess) return e;
        }
        cudaError_t err = cudaSuccess;
        for (int q = 0; q < n && err == cudaSuccess; ++q) {
            cudaStream_t s = n_side > 0 && q % (n_side + 1) ? side->stream[q % (n_side + 1) - 1] : st;
            if (regions[q] == kEvalRest)
                cm_evaluate_list_warp_kernel<T><<<(unsigned)std::min<uint64_t>((round + 3) / 4, 148 * 5), 128, 0, s>>>(t, b, ev);
            else if (regions[q] == kEvalShallow)
                cm_evaluate_list_shallow_kernel<T><<<(unsigned)std::min<uint64_t>((round + 127) / 128, 148 * 4), 128, 0, s>>>(t, b, ev);
            else { err = launch_evaluate_deep(t, b, ev, regions[q], s); continue; }
            err = cudaGetLastError();
        }
        for (int k = 0; k < n_side; ++k) {   // joined even after a failed launch
            cudaError_t j = cudaEventRecord(side->join[k], side->stream[k]);
            if (j == cudaSuccess) j = cudaStreamWaitEvent(st, side->join[k], 0);
            if (err == cudaSuccess) err = j;
        }
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

template <typename T>
static cudaError_t evaluate_space(const Tables &t, const BatchDev &b, const EvalDev &ev, uint64_t stages, uint4 *workspace, cudaStream_t st,
                                  const SideStreams *side) {
    if (!(stages >> kRegStagesMax)) {
        cm_evaluate_shallow_kernel<T><<<(unsigned)((ev.count + 127) / 128), 128, 0, st>>>(t, b, ev);
        return cudaGetLastError();
    }
    // One deep candidate takes a thread ~50 us (its chain of 2 S m cells), a warp ~10; a warp spends five
    // times the instructions, so it is the better one until the warps of a call fill the GPU about twice.
    if (ev.count <= kEvalWarpMax) {
        cm_evaluate_warp_kernel<T><<<(unsigned)((ev.count + 3) / 4), 128, 0, st>>>(t, b, ev);
        return cudaGetLastError();
    }
    return evaluate_binned<T>(t, b, ev, stages, workspace, st, side);
}

cudaError_t launch_evaluate(const Tables &t, const BatchDev &b, EvalDev ev, int single_policy, uint64_t stages, uint4 *workspace,
                            cudaStream_t st, const SideStreams *side) {
    if (ev.count == 0) return cudaSuccess;
    if (single_policy >= 0) {
        cm_evaluate_single_kernel<<<(unsigned)((ev.count + 127) / 128), 128, 0, st>>>(b, ev, single_policy, batch_inf_bits(b));
        return cudaGetLastError();
    }
    return native_i64(b) ? evaluate_space<long long>(t, b, ev, stages, workspace, st, side)
                         : evaluate_space<double>(t, b, ev, stages, workspace, st, side);
}

}  // namespace cm
