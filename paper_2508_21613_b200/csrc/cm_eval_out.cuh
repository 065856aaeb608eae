// Outputs and list entries of cm_evaluate, shared by its kernels (cm_evaluate.cu, cm_cost_impl.cuh).
#pragma once

#include "cm_plan_eval.cuh"

namespace cm {

__device__ __forceinline__ void eval_out_bits(const BatchDev &bd, const EvalDev &ev, uint64_t t, bool ok, uint64_t bits) {
    if (ev.cost && bd.mode == CM_COST_FP64) ev.cost[t] = __longlong_as_double((long long)bits);
    if (ev.cost_ns && bd.mode == CM_COST_INT64NS) ev.cost_ns[t] = batch_cost_ns(bd, bits);
    if (ev.feas) ev.feas[t] = ok ? 1 : 0;
}
template <typename T> __device__ __forceinline__ void eval_out(const BatchDev &bd, const EvalDev &ev, uint64_t t, bool ok, T cost) {
    eval_out_bits(bd, ev, t, ok, Num<T>::bits(cost));
}

__device__ __forceinline__ uint4 *eval_region(const EvalDev &ev, int region) { return ev.list + (size_t)ev.place[region] * ev.slab; }
struct EvalEntry { uint64_t t; SegView g; Cand cand; };
__device__ __forceinline__ EvalEntry eval_entry(const BatchDev &bd, const EvalDev &ev, int region, uint32_t i) {
    const uint4 e = eval_region(ev, region)[i];
    const uint64_t word = (uint64_t)e.z | ((uint64_t)e.w << 32);
    EvalEntry x;
    x.t = ev.base + (e.x & ~kEvalMasked);
    x.g = seg_view(bd, 0, e.y);
    x.cand = e.x & kEvalMasked ? Cand{0, word, 0, true} : Cand{word, 0, 0, false};   // (a masked one is no min-max partition: any rank below K)
    return x;
}

}  // namespace cm
