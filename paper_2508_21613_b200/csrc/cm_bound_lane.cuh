// What the kernels of the bounded search pass (cm_bound.cu, cm_refine.cu) share: a layer composition's
// terms in a lane's registers, the segments of a CTA, the bound of (composition, segment) in floats.
#pragma once

#include "cm_bound.cuh"

namespace cm {

// Bounds of whole buckets are floats rounded down: the per-plan inner loop costs one addition and one
// maximum per stage at full rate (in double arithmetic an addition and a compare-and-select take six
// issue slots).
constexpr float kFloatSlack = 1.0f - 1.0f / (1 << 23);
constexpr float kTieWindow = 1.0f / (1 << 18);     // bounds this close to the least one of a segment are compared bit for bit
constexpr int kBoundThreads = 128;
constexpr float kNoWalk = -__builtin_huge_valf();   // value of a walk that does not exist

struct SegLite {
    uint64_t tier;
    uint64_t lim_bits;   // phase 2: list a plan whose walk costs at most this
    double lim;          // phases 1, 2: look at plans whose bound is at most lim ...
    float ev;            //   ... and above ev (what phase 1 has settled already)
    float coef;          // synchronisation time per gradient byte
    uint32_t scen, tseg, row;
    int n_sync;
};

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
__device__ __forceinline__ SegLite seg_lite(const Tables &tb, const BoundSeg &g) {
    SegLite s;
    s.tier = g.tier; s.scen = g.scen; s.tseg = g.tseg; s.row = g.row; s.n_sync = g.n_sync;
    s.lim = 0.0; s.lim_bits = 0; s.ev = -1.0f;
    s.coef = g.n_sync <= 1 ? 0.0f : __double2float_rd((2.0 * (double)(g.n_sync - 1)) / ((double)g.n_sync * (double)tb.prof->bw_sync));
    return s;
}

// Bucket, tile of compositions and group of segments of a CTA.
struct BoundJob { uint32_t tile, group, s0, s1; uint64_t tile0; };
__device__ __forceinline__ uint32_t bound_bucket(const BoundDev &bo, uint32_t cta) {
    uint32_t lo = 0, hi = bo.n_buckets - 1;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (bo.bucket[mid].chunk_first <= cta) lo = mid; else hi = mid - 1;
    }
    return lo;
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

// Everything a lane knows about its layer composition: b[i] + X_i is the best walk through stage i
// whose visits stay on the cheaper link tier, X_i = 2 * (transfers of boundaries i .. S-2).
template <int NB> struct LaneBound {
    float b[4 * NB];
    float u0, once, g;
    bool ok;
};

// cc / dd (shared memory, a column per thread): stage i's walk with visits upwards / downwards, what
// a boundary on the slower tier adds comes on top.
template <typename T, int NB, bool UNI_X>
__device__ __forceinline__ void lane_setup(LaneBound<NB> &v, const SProf<T> &s, const CutEdges &w, int S, int m, bool check,
                                           float *cc, float *dd, uint8_t *cutc) {
    const bool gpipe = s.sched == CM_SCHED_GPIPE;
    constexpr double none = (double)kNoWalk;
    double U = 0.0, fmax = 0.0, bmax = 0.0;
    double base_n = none, c_n = none, w_n = 0.0, xm_n = 0.0, q_n = 0.0;   // of stage i+1
    long long g_max = 0;
    int hi = s.L;
#pragma unroll
    for (int i = 4 * NB - 1; i >= 0; --i) {
        v.b[i] = kNoWalk;
        if (i < S) {
            const int lo = w.edge(i);
            if (check && (hi <= lo || !stage_fits(s.PS[hi] - s.PS[lo], s.PA[hi] - s.PA[lo], i, S, m, s.cap, s.sched))) v.ok = false;
            const double f = (double)(s.PF[hi] - s.PF[lo]), bk = (double)(s.PB[hi] - s.PB[lo]), wi = f + bk;
            const long long g = s.PP[hi] - s.PP[lo];
            g_max = g > g_max ? g : g_max;
            fmax = tmax(fmax, f);
            bmax = tmax(bmax, bk);
            U += wi;
            if (!gpipe) {
                const bool below_top = i < S - 1;
                const double xm = below_top ? (double)(s.XT[0][hi - 1] < s.XT[1][hi - 1] ? s.XT[0][hi - 1] : s.XT[1][hi - 1]) : 0.0;
                const int n = m - 1 + i - S;
                const double q = n > 1 ? (double)(n >> 1) : 0.0;
                if (below_top) {   // stage i+1 is complete now that its lower neighbour is known
                    const double d = q_n > 0.0 ? base_n + q_n * (wi - w_n) : none;
                    const double best = tmax(base_n, tmax(c_n + 2.0 * q_n * xm_n, d + 2.0 * q_n * xm));
                    if (i + 1 < 4 * NB) v.b[i + 1 < 4 * NB ? i + 1 : 0] = __double2float_rd(best);
                    dd[(i + 1) * kBoundThreads] = __double2float_rd(d);
                }
                base_n = n >= 0 ? U + (double)n * wi : none;
                c_n = q > 0.0 && below_top ? base_n + q * (w_n - wi) : none;
                cc[i * kBoundThreads] = __double2float_rd(c_n);
                w_n = wi; xm_n = xm; q_n = q;
                if (i == 0) v.b[0] = __double2float_rd(tmax(base_n, c_n + 2.0 * q_n * xm_n));
            }
            if (!UNI_X) cutc[i * kBoundThreads] = (uint8_t)hi;
            hi = lo;
        }
    }
    v.u0 = __double2float_rd(U);
    v.once = __double2float_rd((double)(m - 1) * (gpipe ? fmax + bmax : tmax(fmax, bmax)));
    v.g = __ll2float_rd(g_max);
}

// pairs of stays at stage i that visits can replace
__device__ __forceinline__ float stay_pairs(int i, int S, int m) {
    const int n = m - 1 + i - S;
    return n > 1 ? (float)(n >> 1) : 0.0f;
}

// Bound of the lane's composition in one segment.  What a segment adds -- the transfers of its link
// tiers -- is summed once per CTA where the transfer times do not depend on the layer (UNI_X: xr), else
// per plan.  slack: 1 where the synchronisation quotient floors.
template <typename T, int NB, bool UNI_X>
__device__ __forceinline__ float lane_value(const LaneBound<NB> &v, const SProf<T> &sp, int S, int m, const SegLite &sg, const float *xr,
                                            float x1, float slack, const float *cc, const float *dd, const uint8_t *cutc) {
                float best = v.once, x_all;
                const uint64_t tier = sg.tier;
                if (UNI_X) {
                        #pragma unroll
                    for (int k = 0; k < NB; ++k) {
                        const float4 x = reinterpret_cast<const float4 *>(xr)[k];
                        best = fmaxf(best, fmaxf(fmaxf(__fadd_rd(v.b[4 * k], x.x), __fadd_rd(v.b[4 * k + 1], x.y)),
                                                 fmaxf(__fadd_rd(v.b[4 * k + 2], x.z), __fadd_rd(v.b[4 * k + 3], x.w))));
                    }
                    x_all = xr[0];
                    if (sp.sched != CM_SCHED_GPIPE)
                        for (uint64_t t = tier; t; t &= t - 1) {   // visits across an inter-node boundary
                            const int i = __ffsll((long long)t) - 1;
                            best = fmaxf(best, __fadd_rd(cc[i * kBoundThreads], __fmaf_rd(2.0f * stay_pairs(i, S, m), x1, xr[i])));
                            best = fmaxf(best, __fadd_rd(dd[(i + 1) * kBoundThreads],
                                                         __fmaf_rd(2.0f * stay_pairs(i + 1, S, m), x1, i + 1 < S - 1 ? xr[i + 1] : 0.0f)));
                        }
                } else {
                    float X = 0.0f;
    #pragma unroll
                    for (int i = 4 * NB - 1; i >= 0; --i) {
                        if (i < S) {
                            if (i < S - 1) {
                                const bool far = (tier >> i) & 1ull;
                                const float x = __double2float_rd((double)sp.XT[far ? 1 : 0][cutc[i * kBoundThreads] - 1]);
                                const float X_up = X;
                                X = __fadd_rd(X, 2.0f * x);
                                if (far && sp.sched != CM_SCHED_GPIPE) {
                                    best = fmaxf(best, __fadd_rd(cc[i * kBoundThreads], __fmaf_rd(2.0f * stay_pairs(i, S, m), x, X)));
                                    best = fmaxf(best, __fadd_rd(dd[(i + 1) * kBoundThreads], __fmaf_rd(2.0f * stay_pairs(i + 1, S, m), x, X_up)));
                                }
                            }
                            best = fmaxf(best, __fadd_rd(v.b[i], X));
                        }
                    }
                    x_all = X;
                }
                const float lb = __fmaf_rd(v.g, sg.coef, __fadd_rd(__fadd_rd(v.u0, x_all), best));
                return fmaxf(__fmul_rd(__fsub_rd(lb, slack), kFloatSlack), 0.0f);
}

// Transfers above every stage, per segment of the CTA (UNI_X).
template <typename T, int NB>
__device__ __forceinline__ void fill_transfers(float *xs, const SProf<T> &sp, int S, const SegLite *segs, int n_act) {
    const float x0 = __double2float_rd((double)sp.XT[0][0]), x1 = __double2float_rd((double)sp.XT[1][0]);
    for (int s = threadIdx.x; s < n_act; s += kBoundThreads) {
        float X = 0.0f;
        for (int i = 4 * NB - 1; i >= 0; --i) {
            if (i < S - 1) X = __fadd_rd(X, 2.0f * (((segs[s].tier >> i) & 1ull) ? x1 : x0));
            xs[s * 4 * NB + i] = X;
        }
    }
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

// Instantiations of the kernel bodies by stages in fours; a depth in between takes the next one.
constexpr int kBoundNb[] = {4, 9, 16};

}  // namespace cm
