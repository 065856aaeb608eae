// Kernels of the plan search (sm_100a) and their launchers.
//
//   cm_prefix_kernel      per-layer prefix sums and per-boundary transfer times
//   cm_minmax_kernel      min-max contiguous layer partition per (stages, micro-batches)
//   cm_feasible_kernel    memory-feasible layer compositions per (stages, micro-batches), listed once
//   (data rerouting / redundant computation: cm_policy.cu)
//   (the search pass over every pipeline-plan lives in cm_cost.cu)
//   cm_best_split_kernel  best (strategy, micro-batch split) per scenario, the winner decoded
//   (pass 2, the lowest layer composition that meets the winning cost: cm_tiebreak.cu)
//   cm_finalize_kernel    assembles the plans and picks the best policy
//   (per-candidate cost / feasibility for cm_evaluate: cm_evaluate.cu)
#include <algorithm>
#include <atomic>

#include "cm_plan_eval.cuh"
#include "cm_launch.cuh"
#include "cm_split.cuh"

namespace cm {

// ----------------------------------------------------------------------------------
// Prefix sums, accumulated left to right so that every consumer of a stage quantity
// performs the same single subtraction (Section "Estimator": stage time / memory are
// sums over the stage's layers).  One thread per array; the arrays are <= 129 long.
// ----------------------------------------------------------------------------------
__global__ void cm_prefix_kernel(DevProfile *p) {
    const int L = p->L;
    switch (threadIdx.x) {
    // intval: the double arrays carry the integer-nanosecond inputs (sums exact below 2^53)
    case 0: { double a = 0.0; p->PFd[0] = a; for (int l = 0; l < L; ++l) { a = a + (p->intval ? (double)p->fwd_i[l] : p->fwd[l]); p->PFd[l + 1] = a; } break; }
    case 1: { double a = 0.0; p->PBd[0] = a; for (int l = 0; l < L; ++l) { a = a + (p->intval ? (double)p->bwd_i[l] : p->bwd[l]); p->PBd[l + 1] = a; } break; }
    case 2: { int64_t a = 0; p->PFi[0] = a; for (int l = 0; l < L; ++l) { a += p->fwd_i[l]; p->PFi[l + 1] = a; } break; }
    case 3: { int64_t a = 0; p->PBi[0] = a; for (int l = 0; l < L; ++l) { a += p->bwd_i[l]; p->PBi[l + 1] = a; } break; }
    case 4: { int64_t a = 0; p->PA[0] = a; for (int l = 0; l < L; ++l) { a += p->act[l]; p->PA[l + 1] = a; } break; }
    case 5: { int64_t a = 0; p->PS[0] = a; for (int l = 0; l < L; ++l) { a += 2 * p->par[l] + p->opt[l]; p->PS[l + 1] = a; } break; }
    case 6: { int64_t a = 0; p->PP[0] = a; for (int l = 0; l < L; ++l) { a += p->par[l]; p->PP[l + 1] = a; } break; }
    case 7: { int64_t a = 0; p->PW[0] = a; for (int l = 0; l < L; ++l) { a += p->par[l] + p->opt[l]; p->PW[l + 1] = a; } break; }
    default: break;
    }
    for (int l = threadIdx.x; l < L; l += blockDim.x) {
        p->XTd[0][l] = p->intval ? (double)(p->p2p[l] / p->bw_intra) : (double)p->p2p[l] / (double)p->bw_intra;
        p->XTd[1][l] = p->intval ? (double)(p->p2p[l] / p->bw_inter) : (double)p->p2p[l] / (double)p->bw_inter;
        p->XTi[0][l] = p->p2p[l] / p->bw_intra;
        p->XTi[1][l] = p->p2p[l] / p->bw_inter;
    }
}

cudaError_t launch_prefix(DevProfile *prof, cudaStream_t st) {
    cm_prefix_kernel<<<1, 128, 0, st>>>(prof);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Min-max layer partition: D[l][s] = min_k max(D[k][s-1], W(k,l)), W = forward+backward
// time of layers [k,l), only over stages that fit in memory at position s-1.  One CTA
// per (S, m) key; stage columns are swept one after the other, the layers of a column
// go to the warps, the split points k to the lanes, and a warp-shuffle argmin carrying
// (value, k) with the lowest k on ties closes each cell.  Backtracking follows the
// stored argmin, which is the smallest k that attains D[l][s].
// ----------------------------------------------------------------------------------
// a warp per layer of a DP column: 32 warps take the column of a 96-layer model in three sweeps
// (the kernel sits on the path of the first search of a survivor count)
constexpr int kMinmaxThreads = 1024;
template <typename T>
__global__ void __launch_bounds__(kMinmaxThreads) cm_minmax_kernel(Tables tb, const uint32_t *keys, int n_keys) {
    __shared__ T PF[kMaxL + 1], PB[kMaxL + 1];
    __shared__ long long PA[kMaxL + 1], PS[kMaxL + 1];
    __shared__ T D[2][kMaxL + 1];
    __shared__ uint8_t argk[kMaxS + 1][kMaxL + 1];
    const DevProfile *p = tb.prof;
    const int L = p->L;
    const uint32_t key = keys[blockIdx.x];
    const int S = (int)(key >> 16), m = (int)(key & 0xffffu);
    const long long cap = p->cap;
    for (int l = threadIdx.x; l <= L; l += blockDim.x) {
        PF[l] = Num<T>::PF(p)[l];
        PB[l] = Num<T>::PB(p)[l];
        PA[l] = p->PA[l];
        PS[l] = p->PS[l];
        D[0][l] = Num<T>::inf();
        D[1][l] = Num<T>::inf();
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    const T INF = Num<T>::inf();
    for (int s = 1; s <= S; ++s) {
        T *cur = D[s & 1];
        const T *prev = D[(s - 1) & 1];
        for (int l = s + warp; l <= L; l += n_warps) {
            T best = INF;
            int best_k = 0;
            if (s == 1) {
                if (lane == 0 && stage_fits(PS[l] - PS[0], PA[l] - PA[0], 0, S, m, cap, tb.sched))
                    best = (PF[l] - PF[0]) + (PB[l] - PB[0]);
            } else {
                for (int k = s - 1 + lane; k <= l - 1; k += 32) {
                    if (prev[k] == INF) continue;
                    if (!stage_fits(PS[l] - PS[k], PA[l] - PA[k], s - 1, S, m, cap, tb.sched)) continue;
                    T w = (PF[l] - PF[k]) + (PB[l] - PB[k]);
                    T v = tmax(prev[k], w);
                    if (v < best) { best = v; best_k = k; }
                }
            }
            for (int o = 16; o > 0; o >>= 1) {
                T ov = __shfl_xor_sync(0xffffffffu, best, o);
                int ok = __shfl_xor_sync(0xffffffffu, best_k, o);
                if (ov < best || (ov == best && ov != INF && ok < best_k)) { best = ov; best_k = ok; }
            }
            if (lane == 0) {
                cur[l] = best;
                argk[s][l] = (uint8_t)best_k;
            }
        }
        // cells of this column below the first reachable layer stay infinite
        for (int l = threadIdx.x; l < s; l += blockDim.x) cur[l] = INF;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        uint8_t *out = tb.mm_cuts + ((size_t)(S - 1) * tb.mm_stride_m + m) * (kMaxS + 1);
        if (D[S & 1][L] == INF) {
            out[0] = 255;
        } else {
            int l = L;
            out[S] = (uint8_t)L;
            for (int s = S; s >= 2; --s) {
                l = argk[s][l];
                out[s - 1] = (uint8_t)l;
            }
            out[0] = 0;
        }
    }
}

cudaError_t launch_minmax(const Tables &t, const uint32_t *keys_dev, int n_keys, int mode, cudaStream_t st) {
    if (n_keys <= 0) return cudaSuccess;
    if (mode == CM_COST_INT64NS) cm_minmax_kernel<long long><<<n_keys, kMinmaxThreads, 0, st>>>(t, keys_dev, n_keys);
    else cm_minmax_kernel<double><<<n_keys, kMinmaxThreads, 0, st>>>(t, keys_dev, n_keys);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Memory-feasible layer compositions of an (S, m) key, in ascending order (Section
// "Estimator", memory estimator: a stage's peak depends on its layers, its position and the
// micro-batches in flight -- not on the failure scenario, so this is done once per key and
// profile).  One CTA per key walks kappa = 0 .. K-1 in chunks of its size and compacts the
// feasible ranks in order (ballot + prefix over the warps); the min-max partition, candidate
// K, closes the list if a memory-feasible partition exists.
// ----------------------------------------------------------------------------------
constexpr int kFeasThreads = 1024;
__global__ void __launch_bounds__(kFeasThreads) cm_feasible_kernel(Tables tb, int layer_mode, const uint32_t *keys,
                                                                   const uint64_t *Ks, const uint32_t *first,
                                                                   uint32_t *pool, ulonglong2 *masks, uint32_t *count_out,
                                                                   int binom_rows_staged) {
    __shared__ long long PA[kMaxL + 1], PS[kMaxL + 1];
    __shared__ uint32_t warp_cnt[kFeasThreads / 32];
    __shared__ uint32_t running;
    // the rows of the binomial table that unranking reads (n <= stages under the remainder rule,
    // n < layers under the full enumeration), staged once: a rank is unranked through ~S dependent
    // look-ups, and this kernel sits on the path of the first search of a survivor count
    extern __shared__ uint64_t binom_s[];
    const DevProfile *p = tb.prof;
    const int L = p->L;
    for (int q = threadIdx.x; q < binom_rows_staged * (kBinomCols + 1); q += blockDim.x) binom_s[q] = tb.binom[q];
    tb.binom = binom_s;
    const uint32_t key = keys[blockIdx.x];
    const int S = (int)(key >> 16), m = (int)(key & 0xffffu);
    const uint64_t K = Ks[blockIdx.x];
    uint32_t *out = pool + first[blockIdx.x];
    ulonglong2 *out_mask = masks + first[blockIdx.x];
    const long long cap = p->cap;
    for (int l = threadIdx.x; l <= L; l += blockDim.x) { PA[l] = p->PA[l]; PS[l] = p->PS[l]; }
    if (threadIdx.x == 0) running = 0;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint64_t base = 0; base < K; base += kFeasThreads) {
        const uint64_t kappa = base + threadIdx.x;
        bool ok = kappa < K;
        ulonglong2 mask = make_ulonglong2(0, 0);
        if (ok) {
            CutWalker cw;
            make_walker(cw, tb, layer_mode, L, S, Cand{kappa, 0, 0, false}, K, 0);
            mask = make_ulonglong2(cw.a, cw.b);
            int lo = 0;
            for (int i = 0; i < S && ok; ++i) {
                const int hi = cw.next();
                ok = hi > lo && stage_fits(PS[hi] - PS[lo], PA[hi] - PA[lo], i, S, m, cap, tb.sched);
                lo = hi;
            }
        }
        const uint32_t vote = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) warp_cnt[warp] = __popc(vote);
        __syncthreads();
        uint32_t before = running, total = 0;
        for (uint32_t w = 0; w < kFeasThreads / 32; ++w) {
            const uint32_t c = warp_cnt[w];
            if (w < warp) before += c;
            total += c;
        }
        if (ok) {
            const uint32_t at = before + __popc(vote & ((1u << lane) - 1u));
            out[at] = (uint32_t)kappa;
            out_mask[at] = mask;
        }
        __syncthreads();
        if (threadIdx.x == 0) running += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        uint32_t n = running;
        if (tb.mm_cuts[(size_t)tb.mm_slot(S, m) * (kMaxS + 1)] == 0) { out_mask[n] = make_ulonglong2(0, 0); out[n++] = (uint32_t)K; }
        count_out[blockIdx.x] = n;
    }
}

cudaError_t launch_feasible(const Tables &t, int layer_mode, const uint32_t *keys_dev, const uint64_t *K_dev,
                            const uint32_t *first_dev, int n_keys, uint32_t *pool, ulonglong2 *masks, uint32_t *count_dev,
                            cudaStream_t st) {
    if (n_keys <= 0) return cudaSuccess;
    // rows 0 .. 64 (remainder rule: n <= CM_MAX_STAGES) or 0 .. 127 (full enumeration: n < CM_MAX_LAYERS)
    const int rows = std::min(t.binom_rows, layer_mode == CM_LAYERS_REMAINDER ? kMaxS + 1 : kMaxL);
    const size_t smem = (size_t)rows * (kBinomCols + 1) * sizeof(uint64_t);
    static std::atomic<uint64_t> configured{0};   // one bit per device, as for the deep cost kernels
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 64 || !((configured.load(std::memory_order_acquire) >> dev) & 1ull)) {
        cudaError_t e = cudaFuncSetAttribute(cm_feasible_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)((size_t)kMaxL * (kBinomCols + 1) * sizeof(uint64_t)));
        if (e != cudaSuccess) return e;
        if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_release);
    }
    cm_feasible_kernel<<<n_keys, kFeasThreads, smem, st>>>(t, layer_mode, keys_dev, K_dev, first_dev, pool, masks, count_dev, rows);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Segments shared between scenarios (USegDev): one CTA per searched scenario, a thread per
// template segment.  cm_useg_key_kernel finds or claims the slot of the row's tier word in its
// class's table (linear probing, at most as many probes as the table has slots; a table holds
// at least twice the rows of its class) and leaves the lowest row per slot as its
// representative; cm_useg_list_kernel appends every representative to its class's list (the
// order within a class is whatever the atomics give: results do not depend on it) and writes down
// which row is searched for each;
// cm_useg_copy_kernel, after the search pass, gives every other row its representative's minimum.
// ----------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t mix64(uint64_t x) {
    x ^= x >> 30; x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27; x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return (uint32_t)x;
}

// phase 0: the heads of the pair classes; phase 1 (a launch of its own, after phase 0 is complete):
// every other row, which joins a pair it finds in the tables of phase 0 before it is keyed itself
__device__ __forceinline__ uint32_t useg_find(const USegDev &ud, const USegClass &c, unsigned long long tier) {
    uint32_t h = mix64(tier) & c.tab_mask;
    for (uint32_t probe = 0; probe <= c.tab_mask; ++probe) {
        const unsigned long long v = ud.tab[c.tab_first + h];
        if (v == tier) return c.tab_first + h;
        if (v == ~0ull) break;
        h = (h + 1) & c.tab_mask;
    }
    return kNoSegClass;
}

__global__ void __launch_bounds__(128) cm_useg_key_kernel(BatchDev bd, USegDev ud, int phase) {
    const uint32_t scen_id = bd.tmpl_scen[blockIdx.x];
    const Scen sc = bd.scen[scen_id];
    const Tmpl tp = bd.tmpl[sc.tmpl];
    for (uint32_t i = threadIdx.x; i < tp.n_tseg; i += blockDim.x) {
        const uint32_t trow = tp.tseg_first + i, row = sc.seg_base + i;
        const uint32_t ci = ud.tseg_cls[trow];
        if (ci == kNoSegClass || ci == kPartnerSeg) {
            if (phase == 0) ud.slot_of[row] = ci;
            continue;
        }
        if ((ci < ud.n_pair_cls) != (phase == 0)) continue;
        const TSeg g = bd.tseg[trow];
        const unsigned long long tier = cut_bits(bd.cross + sc.cross_first, g.off, g.S - 1);   // < 2^63: never all-ones
        if (phase == 1) {
            uint32_t found = kNoSegClass;
            const uint32_t lh = ud.look_head[trow], lp = ud.look_part[trow];
            if (lh != kNoSegClass) found = useg_find(ud, ud.cls[lh], tier);
            if (found == kNoSegClass && lp != kNoSegClass) {
                found = useg_find(ud, ud.cls[lp], tier);
                if (found != kNoSegClass) found |= kSecondRowFlag;
            }
            if (found != kNoSegClass) { ud.slot_of[row] = found; continue; }
        }
        const USegClass c = ud.cls[ci];
        uint32_t slot = kNoSegClass;
        uint32_t h = mix64(tier) & c.tab_mask;
        for (uint32_t probe = 0; probe <= c.tab_mask; ++probe) {
            const unsigned long long old = atomicCAS(&ud.tab[c.tab_first + h], ~0ull, tier);
            if (old == ~0ull || old == tier) { slot = c.tab_first + h; break; }
            h = (h + 1) & c.tab_mask;
        }
        if (slot == kNoSegClass) atomicAdd(&ud.count[ud.n_cls], 1u);   // (no free slot: cannot happen)
        else atomicMin(&ud.rep[slot], row);
        ud.slot_of[row] = slot;
    }
}

__global__ void __launch_bounds__(128) cm_useg_list_kernel(BatchDev bd, USegDev ud) {
    const uint32_t scen_id = bd.tmpl_scen[blockIdx.x];
    const Scen sc = bd.scen[scen_id];
    const Tmpl tp = bd.tmpl[sc.tmpl];
    for (uint32_t i = threadIdx.x; i < tp.n_tseg; i += blockDim.x) {
        const uint32_t trow = tp.tseg_first + i, row = sc.seg_base + i;
        const uint32_t slot = ud.slot_of[row];
        if (slot == kNoSegClass) { ud.row_rep[row] = row; continue; }
        if (slot == kPartnerSeg) { ud.row_rep[row] = ud.rep[ud.slot_of[row - 1]] + 1; continue; }   // second row of a keyed pair head
        if (slot & kSecondRowFlag) { ud.row_rep[row] = ud.rep[slot & ~kSecondRowFlag] + 1; continue; }
        const uint32_t rep = ud.rep[slot];
        ud.row_rep[row] = rep;
        if (rep != row) continue;
        const uint32_t ci = ud.tseg_cls[trow];   // a representative was keyed in its own class
        const uint32_t pos = atomicAdd(&ud.count[ci], 1u);
        ud.list[ud.cls[ci].list_first + pos] = make_uint2(scen_id, trow);
    }
}

__global__ void __launch_bounds__(256) cm_useg_copy_kernel(BatchDev bd, USegDev ud) {
    const uint32_t row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= bd.n_rows) return;
    const uint32_t r = ud.row_rep[row];
    if (r != row) bd.seg_best[row] = bd.seg_best[r];   // representatives and their second rows are only read here
}

cudaError_t launch_useg_keys(const BatchDev &b, const USegDev &u, cudaStream_t st) {
    if (u.n_rep_scen == 0) return cudaSuccess;
    cm_useg_key_kernel<<<u.n_rep_scen, 128, 0, st>>>(b, u, 0);
    cm_useg_key_kernel<<<u.n_rep_scen, 128, 0, st>>>(b, u, 1);
    cm_useg_list_kernel<<<u.n_rep_scen, 128, 0, st>>>(b, u);
    return cudaGetLastError();
}

cudaError_t launch_useg_copy(const BatchDev &b, const USegDev &u, cudaStream_t st) {
    if (b.n_rows == 0) return cudaSuccess;
    cm_useg_copy_kernel<<<(b.n_rows + 255) / 256, 256, 0, st>>>(b, u);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Best (strategy, micro-batch split) of a scenario: the slowest pipeline's best cost (Section "Estimator":
// step time = max over pipelines), ties to the first strategy and to its split of lowest rank.  A warp per
// strategy; no split is enumerated.
//
// Remainder rule: cm_split.cuh gives the step time; the R larger shares go where they must and then to the
// lowest pipelines that may have them (colexicographic ranks grow with the highest element first).
//
// Full enumeration: a step time t is within reach if shares that every pipeline can take within t add up to
// G, and the least such t is found by halving the range between two costs.  A pipeline's best cost does not
// fall when it gets one more micro-batch, so what it can take is all up to a largest share.  (Costs can fall
// only where the min-max partition is the only candidate and memory forces a luckier one; such a strategy
// is seen, and the sums within reach are kept as a set of bits.)  The split of lowest rank gives the last
// pipelines as many as they can take.
// ----------------------------------------------------------------------------------
// Micro-batches from which halving takes fewer dependent loads than counting up (one failure of the 32-device job,
// three pipelines, 8, 16, 32 and 64 micro-batches: 60, 70, 81 and 110 us a call counting, 64, 73, 79 and 95 halving).
constexpr int kHalveFrom = 32;
struct FullSplit {   // full enumeration, lane = pipeline
    const BatchDev &bd; const Tmpl &tp; const Scen &sc; const Strat &s;
    uint64_t inf;
    __device__ __forceinline__ uint64_t share_cost(int p, int m) const {   // of pipeline p with m micro-batches
        if (m < 1 || m > (int)s.n_m) return inf;
        const uint64_t v = bd.seg_best[canon_row(bd, tp, sc, s, p, m - 1)];
        return v < inf ? v : inf;
    }
    __device__ __forceinline__ uint64_t cost(int m) const {                // of this lane's
        const int lane = threadIdx.x & 31;
        return lane < (int)s.dp ? share_cost(lane, m) : inf;
    }
    __device__ __forceinline__ bool monotone() const {
        bool ok = true;
        for (int q = threadIdx.x & 31; q < (int)s.dp * (int)(s.n_m - 1); q += 32) {
            const int p = q / (s.n_m - 1), k = q - p * (s.n_m - 1);
            const uint64_t a = bd.seg_best[canon_row(bd, tp, sc, s, p, k)], c = bd.seg_best[canon_row(bd, tp, sc, s, p, k + 1)];
            ok = ok && (a < inf ? a : inf) <= (c < inf ? c : inf);
        }
        return __all_sync(0xffffffffu, ok);
    }
    // largest share of this lane's pipeline within t (0: none), costs growing
    __device__ __forceinline__ int most(uint64_t t) const {
        int lo = 0, hi = (threadIdx.x & 31) < (int)s.dp ? (int)s.n_m : 0;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cost(mid) <= t) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
    // Least step time, costs growing.
    __device__ __forceinline__ uint64_t best(int G) const {
        const int lane = threadIdx.x & 31, dp = s.dp;
        // nobody does without a micro-batch, and one pipeline at least takes an equal share or more
        const uint64_t one = ~warp_min_u64(lane < dp ? ~cost(1) : ~0ull), equal = lane < dp ? cost((G + dp - 1) / dp) : inf;
        uint64_t lo = warp_min_u64(equal), hi = ~warp_min_u64(lane < dp ? ~equal : ~0ull);
        lo = one > lo ? one : lo;
        if (dp == 1 || lo >= inf) return lo;
        if (G < kHalveFrom) {                          // everybody takes one more within t, and where nobody can t moves to the least next cost
            uint64_t t = lo;
            int m = most(t), sum = m;
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            uint64_t next = cost(m + 1);
            while (sum < G && t < inf) {
                const uint32_t who = __ballot_sync(0xffffffffu, next <= t);
                if (who) {
                    sum += __popc(who);
                    if (next <= t) next = cost(++m + 1);
                } else {
                    t = warp_min_u64(next);
                }
            }
            return t;
        }
        hi = hi > lo ? hi : lo;
        if (hi >= inf) hi = inf;                       // not known to be within reach
        for (uint64_t t = lo; lo < hi; t = lo + (hi - lo) / 2) {
            const int m = most(t);
            int sum = m;
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (sum >= G) hi = ~warp_min_u64(lane < dp ? ~cost(m) : ~0ull);
            else lo = warp_min_u64(cost(m + 1));
        }
        return hi;
    }
    // The same whatever the costs.  Sums are of shares less one; `sets`: room for two of them (words bits
    // each), `prefix` (or null) for one per pipeline: the sums of the pipelines below it.
    // below, above: the largest cost up to t and the least one above.
    __device__ __forceinline__ bool reach(uint64_t t, int G, int words, uint64_t *sets, uint64_t *prefix, uint64_t &below, uint64_t &above) const {
        const int lane = threadIdx.x & 31;
        uint64_t *now = sets, *next = sets + words, under = 0, over = inf;
        for (int w = lane; w < words; w += 32) now[w] = w == 0 ? 1ull : 0ull;
        __syncwarp();
        for (int p = 0; p < (int)s.dp; ++p) {
            if (prefix)
                for (int w = lane; w < words; w += 32) prefix[p * words + w] = now[w];
            for (int w = lane; w < words; w += 32) next[w] = 0ull;
            __syncwarp();
            for (int base = 0; base < (int)s.n_m; base += 32) {
                const uint64_t c = share_cost(p, base + lane + 1);
                const bool ok = c <= t && c < inf;
                if (ok) under = c > under ? c : under;
                else over = c < over ? c : over;
                if (!__any_sync(0xffffffffu, ok)) continue;
                const int skip = (base + lane) >> 6, bits = (base + lane) & 63;   // this lane's share moves the sums up by
                for (int w = base >> 6; w < words; ++w) {
                    uint64_t v = 0;
                    if (ok && w >= skip) {
                        v = now[w - skip] << bits;
                        if (bits && w > skip) v |= now[w - skip - 1] >> (64 - bits);
                    }
                    const uint32_t v0 = __reduce_or_sync(0xffffffffu, (uint32_t)v), v1 = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
                    if (lane == 0) next[w] |= ((uint64_t)v1 << 32) | v0;
                }
            }
            __syncwarp();
            uint64_t *swap = now; now = next; next = swap;
        }
        below = ~warp_min_u64(~under);
        above = warp_min_u64(over);
        const int goal = G - (int)s.dp;
        const bool got = (now[goal >> 6] >> (goal & 63)) & 1ull;
        __syncwarp();
        return got;
    }
    __device__ __forceinline__ uint64_t best_any(int G, int words, uint64_t *sets) const {
        uint64_t lo = 0, hi, above;
        if (!reach(inf, G, words, sets, nullptr, hi, above)) return inf;
        while (lo < hi) {
            uint64_t below;
            if (reach(lo + (hi - lo) / 2, G, words, sets, nullptr, below, above)) hi = below; else lo = above;
        }
        return hi;
    }
    // micro-batches of this lane's pipeline in the split of lowest rank within t, and that rank
    __device__ __forceinline__ int micro(const uint64_t *binom, int G, uint64_t t, bool growing, int words, uint64_t *sets, uint64_t *prefix,
                                         uint64_t &rank) const {
        const int lane = threadIdx.x & 31, dp = s.dp;
        int left = G, mine = 0, before = 0;
        if (growing) {
            const int can_take = most(t);
            for (int p = dp - 1; p >= 0; --p) {
                const int can = __shfl_sync(0xffffffffu, can_take, p), room = left - p;   // (the p pipelines below get one each at least)
                const int take = can < room ? can : room;
                left -= take;
                if (lane == p) { mine = take; before = left; }                            // before: micro-batches of the pipelines below
            }
        } else {
            uint64_t below, above;
            reach(t, G, words, sets, prefix, below, above);
            left = G - dp;
            for (int p = dp - 1; p >= 0; --p) {
                int take = 0;
                for (int base = ((int)s.n_m - 1) & ~31; base >= 0 && take == 0; base -= 32) {
                    const int m = base + lane + 1, rest = left - (m - 1);
                    const bool ok = m <= (int)s.n_m && rest >= 0 && share_cost(p, m) <= t && ((prefix[p * words + (rest >> 6)] >> (rest & 63)) & 1ull);
                    const uint32_t who = __ballot_sync(0xffffffffu, ok);
                    if (who) take = base + 32 - __clz((int)who);
                }
                left -= take - 1;
                if (lane == p) { mine = take; before = left + p; }
            }
        }
        rank = lane > 0 && lane < dp ? binom_at(binom, before - 1, lane) : 0ull;
        for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        return mine;
    }
};

// win (a search by bounds): the strategies whose step times from bounds are within reach, one of them the best.
// words: 64-bit words of a set of sums (full enumeration); dynamic shared memory: two sets per warp, then one per
// pipeline.
template <bool FULL>
__global__ void __launch_bounds__(1024, 1) cm_best_split_kernel(Tables tb, BatchDev bd, const SearchWin *win, uint64_t inf, int words) {
    extern __shared__ uint64_t sum_sets[];
    __shared__ uint64_t rc[32];
    __shared__ uint32_t ri[32];
    const uint32_t b = blockIdx.x;
    const Scen sc = bd.scen[b];
    const Tmpl tp = bd.tmpl[sc.tmpl];
    const Strat *strat = bd.strat + tp.strat_first;
    const uint32_t warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    const int lane = threadIdx.x & 31, G = tb.prof->G;
    after_previous();
    auto cost_of = [&](const Strat &s) { return strat_cost(bd, tp, sc, s, inf, [&](uint32_t row) { return bd.seg_best[row]; }); };
    uint64_t best_c = inf;
    uint32_t best_i = 0;
    const bool by_list = win && win[b].n_strat <= (uint32_t)kWinStrats;
    const uint32_t n_look = by_list ? win[b].n_strat : tp.n_strat;
    if (sc.rep == b)   // (else it shares another scenario's search: nothing to tie-break here)
        for (uint32_t q = warp; q < n_look; q += warps) {
            const uint32_t si = by_list ? win[b].strat[q] : q;
            const Strat &s = strat[si];
            uint64_t v = inf;
            if constexpr (!FULL) {
                v = strat_best(cost_of(s), s, ~0ull, inf);
            } else if (s.n_m >= 1) {
                const FullSplit fs{bd, tp, sc, s, inf};
                v = fs.monotone() ? fs.best(G) : fs.best_any(G, words, sum_sets + (size_t)warp * 2 * words);
            }
            if (v < best_c || (v == best_c && v < inf && si < best_i)) { best_c = v; best_i = si; }
        }
    if (lane == 0) { rc[warp] = best_c; ri[warp] = best_i; }
    __syncthreads();
    if (warp) return;
    best_c = lane < (int)warps ? rc[lane] : inf;
    best_i = lane < (int)warps ? ri[lane] : 0xffffffffu;
    for (int o = 16; o > 0; o >>= 1) {
        const uint64_t oc = __shfl_xor_sync(0xffffffffu, best_c, o);
        const uint32_t oi = __shfl_xor_sync(0xffffffffu, best_i, o);
        if (oc < best_c || (oc == best_c && oi < best_i)) { best_c = oc; best_i = oi; }
    }
    Winner &w = bd.winner[b];
    uint64_t *kappa = bd.kappa_sel + (size_t)b * kMaxP;
    if (best_c >= inf) {
        if (lane == 0) { w.cost_bits = inf; w.item = ~0ull; w.strat = 0; w.dp = 0; w.scen = b; w.open = 0; }
        if (lane < kMaxP) { w.seg[lane] = 0; w.micro[lane] = 0; kappa[lane] = ~0ull; }
        return;
    }
    const Strat &s = strat[best_i];
    const bool mine = lane < (int)s.dp;                               // lane = pipeline from here on
    int micro;
    uint64_t rank;
    if constexpr (FULL) {
        const FullSplit fs{bd, tp, sc, s, inf};
        micro = fs.micro(tb.binom, G, best_c, fs.monotone(), words, sum_sets, sum_sets + (size_t)warps * 2 * words, rank);
    } else {
        const uint64_t v = cost_of(s);
        const uint64_t lo = __shfl_sync(0xffffffffu, v, (2 * lane) & 31), hi = __shfl_sync(0xffffffffu, v, (2 * lane + 1) & 31);
        const uint32_t must = __ballot_sync(0xffffffffu, mine && lo > best_c);
        const uint32_t may = s.R ? __ballot_sync(0xffffffffu, mine && hi <= best_c) & ~must : 0u;
        const int need = (int)s.R - __popc(must);
        const uint32_t below = (1u << lane) - 1u;
        const bool extra = mine && (((must >> lane) & 1u) || (((may >> lane) & 1u) && __popc(may & below) < need));
        const uint32_t set = __ballot_sync(0xffffffffu, extra);
        rank = extra ? binom_at(tb.binom, lane, __popc(set & below) + 1) : 0ull;
        for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
        micro = mine ? s.m_lo[lane] + (extra ? 1 : 0) : 0;
    }
    if (lane == 0) {
        w.cost_bits = best_c;
        w.item = s.split_first + rank;
        w.strat = tp.strat_first + best_i;
        w.dp = s.dp;
        w.scen = b;
        w.open = 0;
    }
    if (lane < kMaxP) {
        const uint32_t seg = mine ? s.seg_first + lane * s.n_m + (micro - s.m_lo[lane]) : 0u;
        w.seg[lane] = seg;
        w.micro[lane] = mine ? (uint16_t)micro : (uint16_t)0;
        // a segment whose only candidate is the min-max partition has nothing to search (init_kappa_sel)
        kappa[lane] = mine && bd.tseg[seg].K == 0 ? 0ull : ~0ull;
    }
}

cudaError_t launch_split_reduce(const Tables &t, const BatchDev &b, const SearchWin *win, cudaStream_t st) {
    if (b.B <= 0) return cudaSuccess;
    // A warp per strategy, latency of its dependent loads: all strategies at once up to a scenario per SM (64 sets
    // of the 64-device job: 8 us with 1024 threads, 12 with 256, 18 with 128), narrower CTAs beyond (515 sets of
    // the 32-device job: 20 us with 256 threads, 25 with 1024, 26 with 128).  By the list of a search by bounds: 515 sets
    // 17 -> 4 us, 2576 sets 47 -> 13.
    const unsigned threads = b.B <= 148 ? 1024 : 256;
    if (b.batch_mode == CM_BATCH_FULL) {
        const int words = t.binom_rows / 64 + 1;   // (the table has a row per micro-batch of the job at least)
        const size_t bytes = (threads / 32 * 2 + kMaxP) * (size_t)words * sizeof(uint64_t);
        return launch_next(cm_best_split_kernel<true>, b.B, threads, bytes, st, t, b, win, batch_inf_bits(b), words);
    }
    return launch_next(cm_best_split_kernel<false>, b.B, threads, 0, st, t, b, win, batch_inf_bits(b), 0);
}

// ----------------------------------------------------------------------------------
// One scenario handled on its own: clears the result words and fetches the few bytes that say which
// devices failed from the host's pinned memory.  One launch of about 4 us (a read across the bus) in place
// of two copies and a clear; with the plans stored to pinned memory by the last kernel one failure of the
// 256-device job went from 177 to 163 us.
// ----------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) cm_prologue_kernel(uint64_t *words, size_t n_words, const uint32_t *ids_host, uint32_t *ids, int n_ids,
                                                          const uint64_t *bits_host, uint64_t *bits, int n_bits) {
    const size_t at = (size_t)blockIdx.x * 256 + threadIdx.x;
    after_previous();
    if (blockIdx.x == 0) {
        for (int i = threadIdx.x; i < n_ids; i += 256) ids[i] = ids_host[i];
        for (int i = threadIdx.x; i < n_bits; i += 256) bits[i] = bits_host[i];
    }
    for (size_t i = at; i < n_words; i += (size_t)gridDim.x * 256) words[i] = ~0ull;
}

cudaError_t launch_prologue(uint64_t *words, size_t n_words, const uint32_t *ids_host, uint32_t *ids, int n_ids,
                            const uint64_t *bits_host, uint64_t *bits, int n_bits, cudaStream_t st) {
    const size_t ctas = (n_words + 255) / 256;
    cm_prologue_kernel<<<(unsigned)(ctas < 148 ? (ctas ? ctas : 1) : 148), 256, 0, st>>>(words, n_words, ids_host, ids, n_ids, bits_host, bits, n_bits);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------------
// Assemble the per-policy plans and the overall best: least cost, ties to the lowest
// policy id (Algorithm 1 keeps the plan with the least estimated time).  Sixteen threads per plan, one
// per pipeline; four plans per scenario, the last the winner: it goes to the front of the array, the plans
// per policy follow scenario by scenario, so that the host hands both out in one piece each.
// Latency of a few dependent loads: 6 us (a thread per plan walked its pipelines one by one).
// ----------------------------------------------------------------------------------
constexpr int kFinalThreads = 64;   // half of them write a part (FinalPart)
__global__ void __launch_bounds__(kFinalThreads) cm_finalize_kernel(Tables tb, BatchDev bd, FinalPart part, uint64_t inf) {
    const uint32_t b = blockIdx.x;
    const int slot = (threadIdx.x >> 4) + (part == kFinalDyn ? 2 : 0), k = threadIdx.x & 15;
    unsigned long long *tail = reinterpret_cast<unsigned long long *>(bd.plans + (size_t)bd.B * (part == kFinalDyn ? 1 : 4));
    if (b == 0 && threadIdx.x < kCounters && part != kFinalFixed) {
        // work counters ride home behind the plans (they start at all-ones, i.e. -1)
        tail[threadIdx.x] = bd.counters[threadIdx.x] + 1ull;
    }
    const DevProfile *p = tb.prof;
    const Scen sc = bd.scen[b];
    const Winner &w = bd.winner[sc.rep];   // its own search, or the one it shares
    uint64_t cost[3];
    for (int pol = 0; pol < 3; ++pol) {
        const uint64_t c = !(sc.policy_mask & (1u << pol)) || (pol == 2 && part == kFinalFixed) ? inf : pol < 2 ? bd.pol_cost[2 * b + pol] : w.cost_bits;
        cost[pol] = c < inf ? c : inf;
    }
    int pol = slot;
    bool any = true;
    if (slot == 3) {
        pol = 0;
        for (int q = 1; q < 3; ++q)
            if (cost[q] < cost[pol]) pol = q;
        any = cost[pol] < inf;             // (else an empty plan)
    }
    if (part == kFinalDyn && slot == 3) {   // the caller has the plan
        if (k == 0) reinterpret_cast<uint8_t *>(tail + kCounters)[b] = any ? (uint8_t)pol : kNoPolicy;
        return;                             // (its half of the warp)
    }
    const bool dyn = pol == CM_DYNPAR, feasible = cost[pol] < inf, filled = any && (!dyn || feasible);
    const int n = !filled ? 0 : dyn ? (int)w.dp : p->n_dp < kMaxP ? p->n_dp : kMaxP;
    uint64_t kappa = k < n && dyn ? bd.kappa_sel[(size_t)sc.rep * kMaxP + k] : 0ull;
    // (a composition that was not found cannot happen for a feasible winner, but is never handed out as a rank)
    const uint32_t lost = __ballot_sync(part == kFinalDyn ? 0xffffu : 0xffffffffu, kappa == ~0ull) >> (threadIdx.x & 16) & 0xffffu;
    if (kappa == ~0ull) kappa = 0ull;
    cm_plan &out = bd.plans[part == kFinalFixed ? 2 * ((size_t)bd.B + b) + slot : part == kFinalDyn || slot == 3 ? (size_t)b : (size_t)bd.B + 3 * (size_t)b + slot];
    if (k == 0) {
        out.policy = any ? pol : 0;
        out.feasible = feasible && !lost ? 1 : 0;
        out.cost = 0.0;
        out.cost_ns = 0;
        if (feasible) plan_set_cost(out, cost[pol], bd);
        out.strategy = filled && dyn ? w.strat - bd.tmpl[sc.tmpl].strat_first : 0u;
        out.n_pipes = !filled ? 0u : dyn ? w.dp : (uint32_t)p->n_dp;
        out.split_rank = filled && dyn ? w.item - bd.strat[w.strat].split_first : 0ull;
    }
    out.stages[k] = k >= n ? (uint16_t)0 : dyn ? bd.strat[w.strat].S[k]
                    : pol == CM_REDUNDANT && feasible ? bd.rc_stages[b * kMaxP + k] : (uint16_t)p->n_pp;
    out.micro[k] = k >= n ? (uint16_t)0 : dyn ? w.micro[k] : (uint16_t)p->n_micro;
    out.kappa[k] = kappa;
}

cudaError_t launch_finalize(const Tables &t, const BatchDev &b, FinalPart part, cudaStream_t st) {
    if (b.B <= 0) return cudaSuccess;
    const uint64_t inf = batch_inf_bits(b);
    cm_finalize_kernel<<<b.B, part == kFinalAll ? kFinalThreads : kFinalThreads / 2, 0, st>>>(t, b, part, inf);
    return cudaGetLastError();
}

}  // namespace cm
