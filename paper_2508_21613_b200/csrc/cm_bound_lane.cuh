// What the kernels of the bounded search pass (cm_bound.cu, cm_refine.cu) share: a layer composition's terms, a column
// of shared memory that its thread sets up, the segments of a CTA, the bound of (composition, segment) in floats.
#pragma once

#include "cm_bound.cuh"
#include "cm_launch.cuh"

namespace cm {

// Bounds of whole buckets are floats rounded down: the per-plan inner loop costs one look-up, one addition and one
// maximum per dear boundary at full rate (in double arithmetic an addition and a compare-and-select take six
// issue slots).
constexpr float kFloatSlack = 1.0f - 1.0f / (1 << 22);
constexpr float kTieWindow = 1.0f / (1 << 18);     // bounds this close to the least one of a segment are compared bit for bit
constexpr int kBoundThreads = 128;                 // compositions side by side
constexpr float kNoWalk = -__builtin_huge_valf();   // value of a walk that does not exist

// What a CTA keeps of a segment: its link tiers, its row, the synchronisation time per gradient byte.
struct SegLite { uint64_t tier; uint32_t row; float coef; };
constexpr int kDearMax = 6;    // dear boundaries (those on the slower link tier) that are looked up by a list
// Terms of a CTA's compositions: [stages][kBoundThreads + 1] floats (UNI_X) or float2, a column per composition.
// A row is one word longer than the threads, so that lanes with a segment each, which look at different rows of
// one column, use different banks.
constexpr int kTermRow = kBoundThreads + 1;
template <bool UNI_X> constexpr uint32_t kTermSize = UNI_X ? sizeof(float) : sizeof(float2);
constexpr int kBoundSegs = 128;   // segments whose data a CTA holds at a time
static_assert(kBoundSegs == kBoundThreads, "a thread per segment");

__device__ __forceinline__ bool native_i64_dev(const BatchDev &b) { return b.mode == CM_COST_INT64NS && !b.intval; }
__device__ __forceinline__ float lb_of(uint64_t lbarg) { return __uint_as_float((uint32_t)(lbarg >> 32)); }
__device__ __forceinline__ double cost_up(uint64_t bits, bool native) {   // a cost as a double, rounded up
    if (native) return bits >= kInfBitsI64 ? __longlong_as_double((long long)kInfBitsF64) : __ll2double_ru((long long)bits);
    return __longlong_as_double((long long)(bits >= kInfBitsF64 ? kInfBitsF64 : bits));
}

// pick[row]: all-ones = the segment is not needed; kPickWanted = needed, nothing compared yet; otherwise
// the least walk cost of its near-ties above the segment's float bound (saturating) and, in the low
// pick_bits, the position of that plan.
constexpr uint64_t kPickWanted = ~0ull - 1ull;
__device__ __forceinline__ int pick_bits(uint64_t count) { return 64 - __clzll((long long)((count - 1) | 1ull)); }
__device__ __forceinline__ uint64_t pick_base(float lb, bool native) {
    return native ? (uint64_t)(long long)lb : (uint64_t)__double_as_longlong((double)lb);
}
__device__ __forceinline__ uint64_t pick_key(uint64_t bits, uint64_t base, uint64_t pos, int nbits) {
    const uint64_t most = (1ull << (62 - nbits)) - 1ull;   // (below the two marks)
    const uint64_t d = bits > base ? bits - base : 0ull;
    return ((d < most ? d : most) << nbits) | pos;
}

// Segment number q of a bucket.
struct BoundSeg : SegView { uint32_t scen, tseg; };
__device__ __forceinline__ BoundSeg bound_segment(const BatchDev &bd, const BBucket &bk, uint32_t q) {
    BoundSeg v;
    if (bk.tmpl == kSharedBucket) {
        const uint2 p = bd.useg[bk.list_first + q];
        v.scen = p.x;
        v.tseg = p.y + bk.second;
    } else {
        const Tmpl &tp = bd.tmpl[bk.tmpl];
        const uint32_t ti = q / tp.n_scen, si = q - ti * tp.n_scen;
        v.scen = bd.tmpl_scen[tp.scen_first + si];
        v.tseg = bd.bucket_tseg[bk.list_first + ti];
    }
    static_cast<SegView &>(v) = seg_view(bd, v.scen, v.tseg);
    return v;
}
// What the kernels after cm_bound_kernel need to know about a segment of the layout (its number q through all buckets).
__device__ __forceinline__ SegRec seg_record(const BoundSeg &g) { return SegRec{g.tier, g.row, g.scen, g.tseg, g.n_sync}; }

// Bucket, tile of compositions and group of segments of a CTA.
struct BoundJob { uint32_t tile, group, s0, s1; uint64_t tile0; };
// The bucket of CTA number `cta`, into shared memory (all threads).  A thread per bucket where there are enough of them, one
// load deep where halving takes four to seven; beyond that the scan grows with the table and halving does not (passes of a
// batch of the 64-device job: 451 buckets 176 us either way, 944 buckets 472 scanned and 424 halved, 2977 buckets 854 and 611).
constexpr uint32_t kScanBuckets = kBoundThreads;
__device__ __forceinline__ void find_bucket(const BoundDev &bo, uint32_t cta, BBucket *out) {
    if (bo.n_buckets > kScanBuckets) {
        if (threadIdx.x == 0) {
            uint32_t lo = 0, hi = bo.n_buckets - 1;
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (bo.bucket[mid].chunk_first <= cta) lo = mid; else hi = mid - 1;
            }
            *out = bo.bucket[lo];
        }
        return;
    }
    const uint32_t t = threadIdx.x;
    if (t >= bo.n_buckets) return;
    const uint32_t first = bo.bucket[t].chunk_first, next = t + 1 < bo.n_buckets ? bo.bucket[t + 1].chunk_first : bo.n_chunks;
    if (first <= cta && cta < next) *out = bo.bucket[t];
}
__device__ __forceinline__ BoundJob bound_job(const BBucket &bk, uint32_t cta) {
    BoundJob j;
    const uint32_t chunk = cta - bk.chunk_first;
    j.tile = chunk / bk.n_groups;
    j.group = chunk - j.tile * bk.n_groups;
    j.tile0 = (uint64_t)j.tile * bk.width;
    j.s0 = j.group * bk.seg_group;
    j.s1 = j.s0 + bk.seg_group < bk.n_seg ? j.s0 + bk.seg_group : bk.n_seg;
    return j;
}

__device__ __forceinline__ float max3(float a, float b, float c) {   // one instruction
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Stays at stage i in its own walk (negative: the walk does not exist), and the pairs of them that
// visits can replace.
__device__ __forceinline__ int stays(int i, int S, int m) { return m - 1 + i - S; }
__device__ __forceinline__ float stay_pairs(int i, int S, int m) {
    const int n = stays(i, S, m);
    return n > 1 ? (float)(n >> 1) : 0.0f;
}

// Which of the two link tiers is the dearer one, and its boundaries among a segment's S-1.
__device__ __forceinline__ int dear_tier(const Tables &tb) { return tb.prof->bw_inter <= tb.prof->bw_intra ? 1 : 0; }
__device__ __forceinline__ uint64_t dear_bits(uint64_t tier, int dear, int S) {
    return (dear ? tier : ~tier) & ((1ull << (S - 1)) - 1ull);
}
// Transfer times of the boundary after a layer, twice, over the cheaper tier and over the dearer one, rounded either way.
struct Transfers { float lo_rd, lo_ru, hi_rd, hi_ru; };
template <typename T> __device__ __forceinline__ Transfers transfers_at(const SProf<T> &s, int layer, int dear) {
    const double lo = 2.0 * (double)s.XT[dear ^ 1][layer], hi = 2.0 * (double)s.XT[dear][layer];
    return Transfers{__double2float_rd(lo), __double2float_ru(lo), __double2float_rd(hi), __double2float_ru(hi)};
}

// What a lane knows about its layer composition.  With k dear boundaries from stage i upwards (k of their extra
// time Delta each in a transfer up and one down) and P_i the cheap transfers below stage i, the walk through
// stage i has a value b_i - P_i + k Delta, all of it but k a matter of the composition.  As k grows downwards, the best
// of all walks is the best of: max over every i of (b_i - P_i), and for the k-th dear boundary from the top,
// after stage j, max over i <= j of (b_i - P_i), plus k Delta.  (Stages further down have more dear boundaries above
// them than k, and their turn comes with the next one.)  The visits across that boundary at its dear price join
// in: one term per (composition, boundary), and a segment costs one addition and one maximum per dear boundary
// instead of one per stage.
// best: the walks that need no dear boundary; u0: the climb and the drop, the cheap transfers included, and once
// more those that best and the terms are short of.
struct LaneBound {
    float best, u0, g;
    bool ok;
};

// Terms of a composition, stage after stage upwards; the boundary below stage i is complete once the stage is known.
// Transfers that depend on the layer (!UNI_X) bring their Delta along in the terms.
// Double arithmetic is kept to the sums that cancel or grow; what is left is done in floats rounded down,
// and the slowest single forward and backward are compared by the upper halves of their bit patterns.
// Where a stage may outweigh the others (busy) the walks along its whole order count as well, with the dearer
// transfers in what they leave out: one number per lane.
template <typename T, bool UNI_X, bool CUTS>
__device__ __forceinline__ void lane_setup(LaneBound &v, const SProf<T> &s, CutWalker w, int S, int m, bool check, int dear,
                                           unsigned char *term_col, uint8_t *cut_col) {
    const bool gpipe = s.sched == CM_SCHED_GPIPE, busy = s.heavy_stage(S);
    constexpr uint32_t row = kTermRow * kTermSize<UNI_X>;
    const T TF = s.PF[s.L], TB = s.PB[s.L];
    Transfers x = transfers_at(s, 0, dear);           // of the boundary below stage i
    float best = kNoWalk, busy_rel = kNoWalk, busy_best = 0.0f;
    float base_p = kNoWalk, down_p = kNoWalk, q_p = 0.0f;   // of stage i-1: its own walk, the best visit downwards
    double w_p = 0.0, P = 0.0, H = 0.0;               // transfers below stage i, over the cheaper and over the dearer tier
    float P_p = 0.0f;                                 // below stage i-1, rounded up
    int fmax = 0, bmax = 0, lo = 0;
    long long g_max = 0;
    bool ok = true;
#pragma unroll 4
    for (int i = 0; i < S; ++i) {
        const int hi = w.next();
        if (CUTS) cut_col[i * kBoundThreads] = (uint8_t)hi;
        ok = ok && hi > lo;
        if (check && !stage_fits(s.PS[hi] - s.PS[lo], s.PA[hi] - s.PA[lo], i, S, m, s.cap, s.sched)) ok = false;
        const double f = (double)(s.PF[hi] - s.PF[lo]), bk = (double)(s.PB[hi] - s.PB[lo]), wi = f + bk;
        const long long g = s.PP[hi] - s.PP[lo];
        g_max = g > g_max ? g : g_max;
        fmax = max(fmax, __double2hiint(f));
        bmax = max(bmax, __double2hiint(bk));
        if (i > 0) {
            if (!UNI_X) x = transfers_at(s, lo - 1, dear);
            P += 2.0 * (double)s.XT[dear ^ 1][lo - 1];
            H += 2.0 * (double)s.XT[dear][lo - 1];
        }
        const float P_i = __double2float_ru(P);
        float term = kNoWalk;
        if (!gpipe) {
            const int n = stays(i, S, m);
            const float q = stay_pairs(i, S, m);
            const double U = (double)(TF - s.PF[lo]) + (double)(TB - s.PB[lo]), dw = wi - w_p;
            const float base = n >= 0 ? __double2float_rd(__fma_rd((double)n, wi, U)) : kNoWalk;
            const float up = q_p > 0.0f ? __fmaf_rd(q_p, __double2float_rd(dw), base_p) : kNoWalk;
            const float down = q > 0.0f && i > 0 ? __fmaf_rd(q, __double2float_rd(-dw), base) : kNoWalk;
            if (i > 0) {
                best = fmaxf(best, __fsub_rd(max3(base_p, down_p, __fmaf_rd(q_p, x.lo_rd, up)), P_p));
                const float d_ru = __fsub_ru(x.hi_ru, x.lo_rd);
                term = max3(best, __fsub_rd(__fmaf_rd(q_p, x.hi_rd, up), P_p), __fsub_rd(__fsub_rd(__fmaf_rd(q, x.hi_rd, down), P_i), d_ru));
            }
            if (busy) {   // uniform
                const float w_lo = __double2float_rd(wi);
                busy_rel = fmaxf(busy_rel, __fadd_rd(__fmaf_rd((float)m, w_lo, -__double2float_ru(U)), __double2float_rd(H)));
                if (n >= -1)
                    busy_best = fmaxf(busy_best, __fmaf_rd(-(float)(S - 1 - i), __double2float_ru(f < bk ? f : bk), __fmul_rd((float)(m - 1), w_lo)));
            }
            down_p = __fmaf_rd(q, x.lo_rd, down);
            base_p = base; w_p = wi; q_p = q; P_p = P_i;
        }
        if (i > 0) {
            if (UNI_X) *reinterpret_cast<float *>(term_col + (i - 1) * row) = term;
            else *reinterpret_cast<float2 *>(term_col + (i - 1) * row) = make_float2(term, fmaxf(__fsub_rd(x.hi_rd, x.lo_ru), 0.0f));
        }
        lo = hi;
    }
    if (UNI_X) *reinterpret_cast<float *>(term_col + (S - 1) * row) = kNoWalk;   // the row that says nothing
    else *reinterpret_cast<float2 *>(term_col + (S - 1) * row) = make_float2(kNoWalk, 0.0f);
    best = fmaxf(best, __fsub_rd(fmaxf(base_p, down_p), P_p));
    const double f1 = __hiloint2double(fmax, 0), b1 = __hiloint2double(bmax, 0);
    float once = __double2float_rd((double)(m - 1) * (gpipe ? f1 + b1 : tmax(f1, b1)));
    once = max3(once, busy_best, __fsub_rd(busy_rel, __double2float_ru(H)));
    v.best = fmaxf(best, __fsub_rd(once, __double2float_ru(P)));
    v.u0 = __fadd_rd(__double2float_rd((double)TF + (double)TB), __fmul_rd(2.0f, __double2float_rd(P)));
    v.g = __ll2float_rd(g_max);
    if (!ok) v.best = v.u0 = __uint_as_float(0x7f800000u);
    v.ok = ok;
}

// A composition's lane (any: there is one); one that is no plan has an infinite bound.
template <typename T, bool UNI_X, bool CUTS>
__device__ __forceinline__ LaneBound lane_of(const SProf<T> &sp, const Tables &tb, const BatchDev &bd, const BBucket &bk, bool any, const Cand &cand, int dear,
                                             unsigned char *term_col, uint8_t *cut_col) {
    const float none = __uint_as_float(0x7f800000u);
    LaneBound v{none, none, 0.0f, false};
    CutWalker w;
    if (any && make_walker(w, tb, bd.layer_mode, sp.L, bk.S, cand, bk.K, tb.mm_slot(bk.S, bk.m)))
        lane_setup<T, UNI_X, CUTS>(v, sp, w, bk.S, bk.m, bk.feas_first == kNoFeasList, dear, term_col, cut_col);
    if (!v.ok)   // (terms of nothing could be no numbers)
        for (int i = 0; i < bk.S; ++i) {
            if (UNI_X) *reinterpret_cast<float *>(term_col + i * kTermRow * kTermSize<UNI_X>) = kNoWalk;
            else *reinterpret_cast<float2 *>(term_col + i * kTermRow * kTermSize<UNI_X>) = make_float2(kNoWalk, 0.0f);
        }
    return v;
}

// Time that a dear boundary adds to a transfer up and one down, where it does not depend on the layer.
template <typename T> __device__ __forceinline__ float dear_extra(const SProf<T> &s, int dear) {
    const Transfers x = transfers_at(s, 0, dear);
    return fmaxf(__fsub_rd(x.hi_rd, x.lo_ru), 0.0f);
}

__device__ __forceinline__ SegLite seg_lite(uint64_t tier, uint32_t row, int n_sync, long long bw_sync) {
    SegLite s{tier, row, 0.0f};
    if (n_sync > 1) s.coef = __double2float_rd((2.0 * (double)(n_sync - 1)) / ((double)n_sync * (double)bw_sync));
    return s;
}
// What the bound of a plan in a segment takes from it: the synchronisation time per gradient byte, what its dear
// boundaries add to a climb and a drop (UNI_X), and where their terms are in a composition's column, topmost
// first (the rest of the list: the row that says nothing).
struct SegHot { uint64_t bits; float coef, extra; uint32_t off[kDearMax]; int n; };
template <bool UNI_X>
__device__ __forceinline__ SegHot seg_hot(const SegLite &sg, int S, int dear, float delta, bool gpipe) {
    SegHot h;
    h.bits = dear_bits(sg.tier, dear, S);
    h.n = __popcll(h.bits);
    h.coef = sg.coef;
    h.extra = UNI_X ? __fmul_rd((float)h.n, delta) : 0.0f;
    if (UNI_X && gpipe) { h.bits = 0; h.n = 0; }   // (no stays, no visits)
    uint64_t bits = h.bits;
#pragma unroll
    for (int k = 0; k < kDearMax; ++k) {
        const int i = bits ? 63 - __clzll((long long)bits) : S - 1;
        h.off[k] = i * kTermRow * kTermSize<UNI_X>;
        if (bits) bits ^= 1ull << i;
    }
    return h;
}

// Bound of a composition in a segment, without the slack (bound_of).  NF: dear boundaries looked at; -1: as many as
// there are.  (The value does not depend on NF as long as it is enough.)  A value below no zero is made of zeros only;
// rounding down makes -0 of a difference of equals, and the least value is found by its bits.
template <bool UNI_X, int NF>
__device__ __forceinline__ float bound_value(float v_best, float v_u0, float v_g, const unsigned char *term_col, const SegHot &h, float delta) {
    float best = v_best, extra = h.extra;
    float a[NF > 0 ? NF : 1];
    if constexpr (NF > 0) {
#pragma unroll
        for (int k = 0; k < NF; ++k) {
            if constexpr (UNI_X) {
                a[k] = __fadd_rd(*reinterpret_cast<const float *>(term_col + h.off[k]), __fmul_rd((float)(k + 1), delta));
            } else {
                const float2 t = *reinterpret_cast<const float2 *>(term_col + h.off[k]);
                extra = __fadd_rd(extra, t.y);
                a[k] = __fadd_rd(t.x, extra);
            }
        }
#pragma unroll
        for (int k = 0; k + 1 < NF; k += 2) best = max3(best, a[k], a[k + 1]);
        if constexpr (NF & 1) best = fmaxf(best, a[NF - 1]);
    } else if constexpr (NF < 0) {
        int k = 0;
        for (uint64_t bits = h.bits; bits;) {   // four at a time, so that their look-ups are under way together
            float a4[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const bool on = bits != 0;
                const int i = on ? 63 - __clzll((long long)bits) : 0;
                if (on) bits ^= 1ull << i;
                if constexpr (UNI_X) {
                    ++k;
                    a4[u] = __fadd_rd(*reinterpret_cast<const float *>(term_col + i * kTermRow * kTermSize<UNI_X>), __fmul_rd((float)k, delta));
                } else {
                    const float2 t = *reinterpret_cast<const float2 *>(term_col + i * kTermRow * kTermSize<UNI_X>);
                    extra = __fadd_rd(extra, on ? t.y : 0.0f);
                    a4[u] = __fadd_rd(t.x, extra);
                }
                if (!on) a4[u] = kNoWalk;
            }
            best = max3(max3(best, a4[0], a4[1]), a4[2], a4[3]);
        }
    }
    return fmaxf(__fmaf_rd(v_g, h.coef, __fadd_rd(__fadd_rd(v_u0, extra), best)), 0.0f);
}
// The same for a composition per lane and one segment for all of them.
template <bool UNI_X>
__device__ __forceinline__ float bound_value_of(const LaneBound &v, const unsigned char *term_col, const SegHot &h, float delta) {
    return h.n <= 2 ? bound_value<UNI_X, 2>(v.best, v.u0, v.g, term_col, h, delta)
         : h.n <= kDearMax ? bound_value<UNI_X, kDearMax>(v.best, v.u0, v.g, term_col, h, delta)
                           : bound_value<UNI_X, -1>(v.best, v.u0, v.g, term_col, h, delta);
}
// slack: 1 where the synchronisation quotient floors
__device__ __forceinline__ float bound_of(float value, float slack) {
    return fmaxf(__fmul_rd(__fsub_rd(value, slack), kFloatSlack), 0.0f);
}

// Append a plan to a list (any subset of a warp's lanes).
__device__ __forceinline__ void list_append(const BatchDev &bd, const BoundDev &bo, int list, uint32_t scen, uint32_t tseg, uint32_t pos) {
    const uint32_t mates = __match_any_sync(__activemask(), list), lane = threadIdx.x & 31;
    const int lead = __ffs(mates) - 1;
    uint32_t at = 0;
    if ((int)lane == lead) at = atomicAdd(&bo.count[list], (uint32_t)__popc(mates)) + 1u;   // counts start at -1
    at = __shfl_sync(mates, at, lead) + __popc(mates & ((1u << lane) - 1u));
    if (at < bo.list_first[list + 1] - bo.list_first[list]) bo.list[bo.list_first[list] + at] = make_uint4(scen, tseg, pos, 0u);
    else bd.counters[4] = 0ull;   // list full: the host repeats the search without bounds
}

}  // namespace cm
