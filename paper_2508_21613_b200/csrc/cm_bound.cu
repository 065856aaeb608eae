// Bounded search pass (sm_100a): least cost per segment without running the recurrence on every
// pipeline-plan.
//
//   cm_bound_kernel    lower bound of every plan of every segment, the least one per segment
//   cm_window_kernel   per scenario: the step times that can still be the answer, and the segments of
//                      the strategies that can reach them
//   cm_refine_kernel   compares plans whose bounds tie, bit for bit (cm_refine.cu)
//   cm_gather_kernel   lists the most promising plan of every segment needed
//   cm_list_kernel     the recurrence on the listed plans
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
// of k pairs, ub is the k-th best step time.  Batches whose segments are shared between scenarios work
// per segment: lo = nothing, ub = the segment's own result.
#include <algorithm>

#include "cm_bound_lane.cuh"

namespace cm {

// A CTA takes kBoundThreads / W segments side by side, W compositions each (W = a power of two that
// holds the bucket's candidates, at most all threads), and walks its group of segments with the
// composition's terms in registers.
template <typename T, int NB, bool UNI_X>
__device__ void bound_body(const SProf<T> &sp, const Tables &tb, const BatchDev &bd, const BoundDev &bo, const BBucket &bk,
                           uint64_t tile0, const SegLite *segs, int n_seg, unsigned long long *seg_min, unsigned char *dyn) {
    const int S = bk.S, m = bk.m, W = bk.width;
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    const int sub = tid / W, n_sub = kBoundThreads / W;
    float *xs = reinterpret_cast<float *>(dyn);                                            // [n_seg][4 NB] (UNI_X)
    float *cc = reinterpret_cast<float *>(dyn + bo.dyn_cols) + tid;                        // [S][threads]
    float *dd = cc + S * kBoundThreads;
    uint8_t *cutc = dyn + bo.dyn_cols + sizeof(float) * 2 * S * kBoundThreads + tid;
    const float x1 = __double2float_rd((double)sp.XT[1][0]);
    if (UNI_X) fill_transfers<T, NB>(xs, sp, S, segs, n_seg);
    const uint64_t pos = tile0 + (tid & (W - 1));
    LaneBound<NB> v;
    v.ok = pos < bk.count;
    if (v.ok) {
        CutWalker w;
        v.ok = make_walker(w, tb, bd.layer_mode, sp.L, S, walk_kappa(bd.feas, bk.feas_first, pos), bk.K, tb.mm_slot(S, m));
        if (v.ok) lane_setup<T, NB, UNI_X>(v, sp, cut_edges(w), S, m, bk.feas_first == kNoFeasList, cc, dd, cutc);
    }
    const int n_ok = __syncthreads_count(v.ok && sub == 0);
    if (tid == 0 && n_ok) {   // what this pass decides: the plans, and the cells recurrences over them would take
        const unsigned long long plans = (unsigned long long)n_ok * (unsigned long long)n_seg;
        const unsigned long long cells = bk.role == 2 ? 0ull
            : bk.role == 1 ? 2ull * S * (m + 1) + 3ull * S * (S - 1) / 2 : 2ull * S * m;
        atomicAdd(&bd.counters[0], plans * cells);
        atomicAdd(&bd.counters[2], plans);
    }
    const float slack = sp.intval || std::is_same<T, long long>::value ? 1.0f : 0.0f;
    const int n_it = (n_seg + n_sub - 1) / n_sub;
    for (int it = 0; it < n_it; ++it) {
        const int s = it * n_sub + sub;
        const bool have = s < n_seg && v.ok;
        float lb = __uint_as_float(0x7f800000u);
        if (have) lb = lane_value<T, NB, UNI_X>(v, sp, S, m, segs[s], xs + s * 4 * NB, x1, slack, cc, dd, cutc);
        if (W >= 32) {   // (the lanes of a warp share the segment)
            const uint32_t mine = __float_as_uint(lb), least = __reduce_min_sync(0xffffffffu, mine);
            const uint32_t who = __ballot_sync(0xffffffffu, mine == least);
            if (have && lane == (uint32_t)(__ffs(who) - 1))
                atomicMin(&seg_min[s], ((unsigned long long)mine << 32) | (uint32_t)pos);
        } else {
            unsigned long long key = have ? ((unsigned long long)__float_as_uint(lb) << 32) | (uint32_t)pos : ~0ull;
            for (int o = W >> 1; o > 0; o >>= 1) {
                const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
                key = k2 < key ? k2 : key;
            }
            if (s < n_seg && (tid & (W - 1)) == 0 && key != ~0ull) seg_min[s] = key;   // the only writer of its segment
        }
    }
}

template <typename T, bool UNI_X>
__global__ void __launch_bounds__(kBoundThreads) cm_bound_kernel(Tables tb, BatchDev bd, BoundDev bo) {
    __shared__ SProf<T> sp;
    __shared__ BBucket bks;
    extern __shared__ __align__(16) unsigned char dyn[];
    const uint32_t tid = threadIdx.x;
    if (tid == 0) bks = bo.bucket[bound_bucket(bo, blockIdx.x)];
    stage_profile(sp, tb);
    __syncthreads();
    const BBucket &bk = bks;
    const BoundJob job = bound_job(bk, blockIdx.x);
    SegLite *segs = reinterpret_cast<SegLite *>(dyn + bo.dyn_segs);
    unsigned long long *seg_min = reinterpret_cast<unsigned long long *>(dyn + bo.dyn_segs + sizeof(SegLite) * bo.max_group);
    const int n_seg = (int)(job.s1 - job.s0);
    for (int q = tid; q < n_seg; q += kBoundThreads) {
        segs[q] = seg_lite(tb, bound_segment(bd, bk, job.s0 + q));
        seg_min[q] = ~0ull;
    }
    __syncthreads();
    const int nb = (bk.S + 3) >> 2;
#define CM_NB(K) if (nb <= K) bound_body<T, K, UNI_X>(sp, tb, bd, bo, bk, job.tile0, segs, n_seg, seg_min, dyn); else
    if constexpr (UNI_X && std::is_same<T, double>::value) { CM_NB(1) CM_NB(2) CM_NB(3) CM_NB(4) CM_NB(6) CM_NB(8) CM_NB(9) CM_NB(12) CM_NB(16) {} }
    else { CM_NB(4) CM_NB(9) CM_NB(16) {} }
#undef CM_NB
    __syncthreads();
    for (int q = tid; q < n_seg; q += kBoundThreads)
        if (seg_min[q] < bo.lbarg[segs[q].row]) atomicMin((unsigned long long *)&bo.lbarg[segs[q].row], seg_min[q]);
}

size_t bound_dyn_bytes(BoundDev &bo, int max_stages, int max_group, bool uniform_x) {
    size_t nb = (size_t)(max_stages + 3) / 4;
    for (size_t k : kBoundNb)
        if (nb <= k) { nb = k; break; }
    size_t off = uniform_x ? (size_t)max_group * 16 * nb : 0;
    bo.dyn_cols = (uint32_t)off;
    off += sizeof(float) * 2 * max_stages * kBoundThreads + (uniform_x ? 0 : (size_t)max_stages * kBoundThreads);
    off = (off + 15) & ~(size_t)15;
    bo.dyn_segs = (uint32_t)off;
    bo.max_group = (uint32_t)max_group;
    return off + (size_t)max_group * (sizeof(SegLite) + sizeof(unsigned long long));
}

template <typename T, bool UNI_X>
static cudaError_t launch_bound_one(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(cm_bound_kernel<T, UNI_X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBoundDynMax);
    if (e != cudaSuccess) return e;
    cm_bound_kernel<T, UNI_X><<<bo.n_chunks, kBoundThreads, bo.dyn_bytes, st>>>(t, b, bo);
    return cudaGetLastError();
}
cudaError_t launch_bound(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    if (bo.n_chunks == 0) return cudaSuccess;
    if (native_i64(b)) return bo.uniform_x ? launch_bound_one<long long, true>(t, b, bo, st) : launch_bound_one<long long, false>(t, b, bo, st);
    return bo.uniform_x ? launch_bound_one<double, true>(t, b, bo, st) : launch_bound_one<double, false>(t, b, bo, st);
}

// ----------------------------------------------------------------------------------
// Window of a scenario under the remainder rule: a strategy hands one more micro-batch to R of its
// pipelines, every choice of them a split, so its best step time is the least value t among its
// pipelines' two costs such that those that cannot do with their smaller share (cost above t) number
// at most R, all pipelines that can take the larger one (cost at most t) number at least R, and the
// former are among the latter; C(may - must, R - must) splits then stay within t.  A thread per
// strategy; phase 0 works on the bounds, phase 1 on the results.  Either then marks the segments of the
// strategies whose step time from bounds is still within reach.
// ----------------------------------------------------------------------------------
struct StratCosts { uint64_t lo[kMaxP], hi[kMaxP]; int dp, R; };
// Phase 0 marks strategies this far above the best step time from bounds: one plan of each of their
// segments is evaluated, so that a result that misses its bound a little still leaves phase 2 nothing to do.
constexpr float kReach = 1.0f / (1 << 13);

__device__ __forceinline__ uint32_t canon_row(const BatchDev &bd, const Tmpl &tp, const Scen &sc, const Strat &s, int p, int k) {
    uint32_t t = s.seg_first + p * s.n_m + k;
    if (bd.tseg_canon) t = bd.tseg_canon[t];
    return sc.seg_base + (t - tp.tseg_first);
}

__device__ __forceinline__ void strat_costs(const BatchDev &bd, const BoundDev &bo, const Tmpl &tp, const Scen &sc, uint32_t si, int phase,
                                            uint64_t inf, StratCosts &c) {
    const Strat &s = bd.strat[tp.strat_first + si];
    c.dp = s.dp;
    c.R = s.R;
    for (int p = 0; p < s.dp; ++p)
        for (int k = 0; k < 2; ++k) {
            uint64_t v = inf;
            if (k < s.n_m && s.m_lo[p] + k >= 1) {
                const uint32_t row = canon_row(bd, tp, sc, s, p, k);
                v = phase ? bd.seg_best[row] : (uint64_t)(bo.lbarg[row] >> 32);
                v = v > inf ? inf : v;
            }
            (k ? c.hi : c.lo)[p] = v;
        }
}

__device__ __forceinline__ bool splits_within(const StratCosts &c, uint64_t t, int &free_ones, int &left) {
    int may = 0, must = 0;
    bool ok = true;
    for (int p = 0; p < c.dp; ++p) {
        const bool can = c.hi[p] <= t, need = c.lo[p] > t;
        may += can;
        must += need;
        ok = ok && (can || !need);
    }
    free_ones = may - must;
    left = c.R - must;
    return ok && left >= 0 && may >= c.R;
}

__device__ __forceinline__ uint64_t strat_best(const StratCosts &c, uint64_t after, uint64_t inf) {   // least t > after (after = ~0: any)
    uint64_t best = inf;
    int f, l;
    for (int p = 0; p < c.dp; ++p)
        for (int k = 0; k < 2; ++k) {
            const uint64_t t = k ? c.hi[p] : c.lo[p];
            if (t < best && (after == ~0ull || t > after) && splits_within(c, t, f, l)) best = t;
        }
    return best;
}

constexpr int kWinThreads = 128;
__device__ __forceinline__ uint64_t block_min_u64(uint64_t v, uint64_t *red) {
    v = warp_min_u64(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    for (int w = 0; w < kWinThreads / 32; ++w) v = red[w] < v ? red[w] : v;
    return v;
}

__global__ void __launch_bounds__(kWinThreads) cm_window_kernel(Tables tb, BatchDev bd, BoundDev bo, int phase, int k_best, uint64_t inf_cost) {
    __shared__ uint64_t red[kWinThreads / 32];
    __shared__ unsigned long long total;
    const uint32_t b = blockIdx.x;
    const Scen sc = bd.scen[b];
    const Tmpl tp = bd.tmpl[sc.tmpl];
    const uint64_t inf = phase ? inf_cost : 0xffffffffull;
    uint64_t first = ~0ull, t = ~0ull;
    bool enough = false;
    for (int r = 0; r < k_best && !enough; ++r) {
        uint64_t mine = inf;
        for (uint32_t si = threadIdx.x; si < tp.n_strat; si += kWinThreads) {
            StratCosts c;
            strat_costs(bd, bo, tp, sc, si, phase, inf, c);
            const uint64_t v = strat_best(c, t, inf);
            mine = v < mine ? v : mine;
        }
        t = block_min_u64(mine, red);
        if (r == 0) first = t;
        if (t >= inf || k_best == 1) break;
        if (threadIdx.x == 0) total = 0;
        __syncthreads();
        unsigned long long n = 0;
        for (uint32_t si = threadIdx.x; si < tp.n_strat; si += kWinThreads) {
            StratCosts c;
            int f, l;
            strat_costs(bd, bo, tp, sc, si, phase, inf, c);
            if (splits_within(c, t, f, l)) n += binom_at(tb.binom, f, l);
        }
        if (n) atomicAdd(&total, n);
        __syncthreads();
        enough = total >= (unsigned long long)k_best;
        __syncthreads();
    }
    if (k_best > 1 && !enough && t < inf) t = inf;
    float reach = -1.0f;   // step times from bounds up to here (-1: none)
    if (phase) {
        if (t < ~0ull) reach = __double2float_ru(cost_up(t, native_i64_dev(bd)));
        if (threadIdx.x == 0) bo.win[b].ub = t;
    } else {
        const float lo = first < inf ? __uint_as_float((uint32_t)first) : 0.0f;
        if (first < inf) reach = t < inf ? __fmul_ru(__uint_as_float((uint32_t)t), 1.0f + kReach) : __uint_as_float(0x7f800000u);
        if (threadIdx.x == 0) bo.win[b] = SearchWin{lo, 0.0f, inf_cost};
    }
    for (uint32_t si = threadIdx.x; si < tp.n_strat; si += kWinThreads) {
        StratCosts c;
        strat_costs(bd, bo, tp, sc, si, 0, 0xffffffffull, c);
        const uint64_t v = strat_best(c, ~0ull, 0xffffffffull);
        if (v >= 0xffffffffull || __uint_as_float((uint32_t)v) > reach) continue;
        const Strat &s = bd.strat[tp.strat_first + si];
        for (int p = 0; p < s.dp; ++p)
            for (int k = 0; k < s.n_m; ++k) {
                const uint32_t row = canon_row(bd, tp, sc, s, p, k);
                if (bo.pick[row] == ~0ull) bo.pick[row] = kPickWanted;   // (every writer writes the same)
            }
    }
}

cudaError_t launch_window(const Tables &t, const BatchDev &b, const BoundDev &bo, int phase, int k_best, cudaStream_t st) {
    if (b.B <= 0) return cudaSuccess;
    cm_window_kernel<<<b.B, kWinThreads, 0, st>>>(t, b, bo, phase, k_best, batch_inf_bits(b));
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// The plan that phase 1 takes per segment: a thread per searched segment.
// ----------------------------------------------------------------------------------
__global__ void __launch_bounds__(128) cm_gather_kernel(Tables tb, BatchDev bd, BoundDev bo) {
    const uint32_t at = blockIdx.x * 128 + threadIdx.x;
    if (at >= bo.n_segs) return;
    uint32_t lo = 0, hi = bo.n_buckets - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (bo.bucket[mid].seg_first <= at) lo = mid; else hi = mid - 1;
    }
    const BBucket bk = bo.bucket[lo];
    const BoundSeg g = bound_segment(bd, bk, at - bk.seg_first);
    const uint64_t la = bo.lbarg[g.row], key = bo.pick[g.row];
    if (la == ~0ull || key == ~0ull) return;   // nothing fits in memory / not needed
    const uint32_t pos = key == kPickWanted ? (uint32_t)la : (uint32_t)(key & ((1ull << pick_bits(bk.count)) - 1ull));
    list_append(bd, bo, bk.S <= kRegStagesMax ? 0 : 1, g.scen, g.tseg, pos);
}

cudaError_t launch_gather(const Tables &t, const BatchDev &b, const BoundDev &bo, cudaStream_t st) {
    if (bo.n_segs == 0) return cudaSuccess;
    cm_gather_kernel<<<(bo.n_segs + 127) / 128, 128, 0, st>>>(t, b, bo);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// The recurrence on the listed plans.  Pipelines of at most 16 stages: a thread per plan, state in
// registers; deeper ones: a warp per plan in lock step, 2(S+m) slots of ~45 cycles (a thread would
// need ~100 us for its chain of 2 S m cells, and the lists are short).  Even CTAs take the shallow
// list, odd ones the deep one.
// ----------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(kChunk) cm_list_kernel(Tables tb, BatchDev bd, BoundDev bo, int first_list) {
    __shared__ SProf<T> sp;
    __shared__ uint8_t cuts_s[kChunk / 32][kMaxS + 8];
    const bool deep = blockIdx.x & 1;
    const uint32_t cta = blockIdx.x >> 1, ctas = gridDim.x >> 1;
    const int list = first_list + (deep ? 1 : 0);
    const uint32_t room = bo.list_first[list + 1] - bo.list_first[list];
    uint32_t n = bo.count[list] + 1u;
    n = n < room ? n : room;
    const uint32_t per = deep ? kChunk / 32 : kChunk;
    if ((uint64_t)cta * per >= n) return;
    stage_profile(sp, tb);
    __syncthreads();
    const uint4 *entries = bo.list + bo.list_first[list];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long work = 0;   // cells in the low 40 bits, plans above
    for (uint32_t i = cta * per + (deep ? warp : threadIdx.x); i < n; i += ctas * per) {
        const uint4 e = entries[i];
        const SegView g = seg_view(bd, e.x, e.y);
        const uint64_t kappa = walk_kappa(bd.feas, g.feas_first, e.z);
        T cost;
        bool ok;
        if (deep) ok = warp_plan_cost<T>(sp, tb, bd.layer_mode, g, kappa, cuts_s[warp], cost);
        else if (g.m >= g.S - 1) ok = plan_cost_regs_any<T>(sp, tb, bd.layer_mode, g, kappa, cost);
        else ok = plan_cost_regs_any<T, true>(sp, tb, bd.layer_mode, g, kappa, cost);
        if (deep && lane) continue;
        if (ok) {
            const uint64_t bits = Num<T>::bits(cost);
            if (bits < bd.seg_best[g.row]) atomicMin((unsigned long long *)&bd.seg_best[g.row], (unsigned long long)bits);
        }
        work += 2ull * g.S * g.m + (1ull << 40);
    }
    for (int o = 16; o > 0; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
    if (lane == 0 && work) {
        atomicAdd(&bd.counters[3], work & ((1ull << 40) - 1ull));
        atomicAdd(&bd.counters[5], work >> 40);
    }
}

cudaError_t launch_list(const Tables &t, const BatchDev &b, const BoundDev &bo, int first_list, uint64_t most, cudaStream_t st) {
    const unsigned grid = 2 * (unsigned)std::min<uint64_t>(std::max<uint64_t>((most + 3) / 4, 1), 148 * 6);
    if (native_i64(b)) cm_list_kernel<long long><<<grid, kChunk, 0, st>>>(t, b, bo, first_list);
    else cm_list_kernel<double><<<grid, kChunk, 0, st>>>(t, b, bo, first_list);
    return cudaGetLastError();
}

}  // namespace cm
