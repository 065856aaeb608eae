// What the kernels of the bounded search pass (cm_bound.cu, cm_refine.cu) share: a layer composition's
// terms in a lane's registers, the segments of a CTA, the bound of (composition, segment) in floats.
#pragma once

#include "cm_bound.cuh"

namespace cm {

// Bounds of whole buckets are floats rounded down: the per-plan inner loop costs one addition and one
// maximum per stage at full rate (in double arithmetic an addition and a compare-and-select take six
// issue slots).
constexpr float kFloatSlack = 1.0f - 1.0f / (1 << 22);
constexpr float kTieWindow = 1.0f / (1 << 18);     // bounds this close to the least one of a segment are compared bit for bit
constexpr int kBoundThreads = 128;
constexpr float kNoWalk = -__builtin_huge_valf();   // value of a walk that does not exist

// What the bound of a segment needs: its link tiers, its row, the synchronisation time per gradient byte,
// how many of its inter-node boundaries are in the list of visits (kFarLong: too many, see lane_value).
struct SegLite { uint64_t tier; uint32_t row; float coef; int n_sync, n_far; };
// A visit across an inter-node boundary between stages `at` and at+1: what it adds to the lane's terms.
struct FarVisit { float up, down; int at, pad; };
constexpr int kFarMax = 6, kFarLong = kFarMax + 1;
// Shared memory of a bound CTA, in this order: transfers above every stage [group][4 NB] floats (UNI_X) |
// visits [group][kFarMax] (UNI_X) | visit terms [stages][threads] float2 | cuts [stages][threads] bytes |
// segments [group] | a 64-bit word per segment | what else the kernel keeps per segment.
struct BoundSmem {
    float *xs;
    FarVisit *far;
    float2 *cd;       // this thread's column
    uint8_t *cut;     // this thread's column
    SegLite *segs;
    unsigned long long *word;
    unsigned char *rest;
};
__device__ __forceinline__ BoundSmem bound_smem(unsigned char *dyn, const BoundDev &bo) {
    BoundSmem m;
    m.xs = reinterpret_cast<float *>(dyn);
    m.far = reinterpret_cast<FarVisit *>(dyn + bo.dyn_far);
    m.cd = reinterpret_cast<float2 *>(dyn + bo.dyn_cols) + threadIdx.x;
    m.cut = dyn + bo.dyn_cuts + threadIdx.x;
    m.segs = reinterpret_cast<SegLite *>(dyn + bo.dyn_segs);
    m.word = reinterpret_cast<unsigned long long *>(dyn + bo.dyn_segs + sizeof(SegLite) * bo.max_group);
    m.rest = reinterpret_cast<unsigned char *>(m.word + bo.max_group);
    return m;
}

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
    SegLite s{g.tier, g.row, 0.0f, g.n_sync, 0};
    if (g.n_sync > 1) s.coef = __double2float_rd((2.0 * (double)(g.n_sync - 1)) / ((double)g.n_sync * (double)tb.prof->bw_sync));
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

// Maximum of three and two additions (rounded down) in one instruction each.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float2 add2_rd(float2 a, float2 b) {
    uint64_t x, y, z;
    float2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
    asm("mov.b64 %0, {%1, %2};" : "=l"(y) : "f"(b.x), "f"(b.y));
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(z) : "l"(x), "l"(y));
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(z));
    return r;
}

// Everything a lane knows about its layer composition: b[i] + X_i is the best walk through stage i
// whose visits stay on the cheaper link tier, X_i = 2 * (transfers of boundaries i .. S-2).
template <int NB> struct LaneBound {
    float2 b[2 * NB];
    float u0, once, g;
    bool ok;
    __device__ __forceinline__ float get(int i) const { return i & 1 ? b[i >> 1].y : b[i >> 1].x; }
    __device__ __forceinline__ void set(int i, float v) { if (i & 1) b[i >> 1].y = v; else b[i >> 1].x = v; }
};

// Stays at stage i in its own walk (negative: the walk does not exist), and the pairs of them that
// visits can replace.
__device__ __forceinline__ int stays(int i, int S, int m) { return m - 1 + i - S; }
__device__ __forceinline__ float stay_pairs(int i, int S, int m) {
    const int n = stays(i, S, m);
    return n > 1 ? (float)(n >> 1) : 0.0f;
}

// cd (shared memory, a column per thread): entry i = the walks that visit across boundary i, from stage i
// upwards and from stage i+1 downwards, without the boundary's transfers.
//
// This is a third of the kernel's instructions, so double arithmetic is kept to the sums that cancel or
// grow (six operations a stage); what is left is done in floats rounded down, and the slowest single
// forward and backward are compared by the upper halves of their bit patterns.
// The stages are a loop of four at a time whose results move up the registers: all of them in a row are
// tens of kilobytes of code per depth that every CTA runs through once, and the warps waited for
// instructions most of the time.  (The whole call changes by less than its runs differ: 1024 sets of the
// 256-device job 2.0 ms either way.)
// Where a stage may outweigh the others (busy) the walks along its whole order count as well.  Their values
// depend on the link tiers through the boundaries that they leave out; with the dearer tier there they are one
// number per lane.
template <typename T, int NB, bool UNI_X>
__device__ __forceinline__ void lane_setup(LaneBound<NB> &v, const SProf<T> &s, const CutColumn<kBoundThreads> &w, int S, int m, bool check, float2 *cd) {
    const bool gpipe = s.sched == CM_SCHED_GPIPE, busy = s.heavy_stage(S);
    float busy_best = 0.0f, U_hi = 0.0f;              // U_hi: U_i with the dearer transfers, rounded up
    double U = 0.0, w_n = 0.0;                        // w_n: of stage i+1
    float base_n = kNoWalk, c_n = kNoWalk, xq_n = 0.0f, q_n = 0.0f;
    const float xm_all = __double2float_rd((double)(s.XT[0][0] < s.XT[1][0] ? s.XT[0][0] : s.XT[1][0]));
    int fmax = 0, bmax = 0;
    long long g_max = 0;
    int hi = s.L;
#pragma unroll
    for (int j = 0; j < 2 * NB; ++j) v.b[j] = make_float2(kNoWalk, kNoWalk);
#pragma unroll 1
    for (int k = (S - 1) >> 2; k >= 0; --k) {   // four stages a turn, topmost first
#pragma unroll
        for (int r = 3; r >= 0; --r) {
            const int i = 4 * k + r;
            if (i < S) {
                const int lo = w.edge(i);
                if (check && (hi <= lo || !stage_fits(s.PS[hi] - s.PS[lo], s.PA[hi] - s.PA[lo], i, S, m, s.cap, s.sched))) v.ok = false;
                const double f = (double)(s.PF[hi] - s.PF[lo]), bk = (double)(s.PB[hi] - s.PB[lo]), wi = f + bk;
                const long long g = s.PP[hi] - s.PP[lo];
                g_max = g > g_max ? g : g_max;
                fmax = max(fmax, __double2hiint(f));
                bmax = max(bmax, __double2hiint(bk));
                U += wi;
                if (!gpipe) {
                    const int n = stays(i, S, m);
                    const float q = stay_pairs(i, S, m);
                    float xm = xm_all, d = kNoWalk;
                    if (!UNI_X) xm = __double2float_rd((double)(s.XT[0][hi - 1] < s.XT[1][hi - 1] ? s.XT[0][hi - 1] : s.XT[1][hi - 1]));
                    const double dw = wi - w_n;
                    if (i < S - 1) {   // stage i+1 is complete now that its lower neighbour is known
                        if (q_n > 0.0f) d = __fmaf_rd(q_n, __double2float_rd(dw), base_n);
                        const float up = c_n == kNoWalk ? kNoWalk : __fadd_rd(c_n, xq_n);
                        v.set(r == 3 ? 0 : r + 1, max3(base_n, up, __fmaf_rd(2.0f * q_n, xm, d)));   // (r == 3: not shifted yet)
                    }
                    base_n = n >= 0 ? __double2float_rd(__fma_rd((double)n, wi, U)) : kNoWalk;
                    c_n = q > 0.0f && i < S - 1 ? __fmaf_rd(q, __double2float_rd(-dw), base_n) : kNoWalk;
                    cd[i * kBoundThreads] = make_float2(c_n, d);
                    w_n = wi; q_n = q; xq_n = __fmul_rd(2.0f * q, xm);
                    if (busy) {   // uniform
                        const int at = UNI_X ? 0 : hi - 1;
                        const float w_lo = __double2float_rd(wi), x_hi = i < S - 1 ? __double2float_ru((double)tmax(s.XT[0][at], s.XT[1][at])) : 0.0f;
                        U_hi = __fadd_ru(U_hi, __fmaf_ru(2.0f, x_hi, __double2float_ru(wi)));
                        busy_best = fmaxf(busy_best, __fmaf_rd((float)m, w_lo, -U_hi));
                        if (n >= -1)
                            busy_best = fmaxf(busy_best, __fmaf_rd(-(float)(S - 1 - i), __double2float_ru(f < bk ? f : bk), __fmul_rd((float)(m - 1), w_lo)));
                    }
                }
                hi = lo;
            }
            if (r == 3) {   // the stages so far move up by four
#pragma unroll
                for (int j = 2 * NB - 1; j > 1; --j) v.b[j] = v.b[j - 2];
                v.b[0] = v.b[1] = make_float2(kNoWalk, kNoWalk);
            }
        }
    }
    if (!gpipe) v.set(0, fmaxf(base_n, c_n == kNoWalk ? kNoWalk : __fadd_rd(c_n, xq_n)));
    const double f1 = __hiloint2double(fmax, 0), b1 = __hiloint2double(bmax, 0);
    v.u0 = __double2float_rd(U);
    v.once = fmaxf(__double2float_rd((double)(m - 1) * (gpipe ? f1 + b1 : tmax(f1, b1))), busy_best);
    v.g = __ll2float_rd(g_max);
}

// Transfers above every stage and the visits across inter-node boundaries, per segment of the CTA, where
// the transfer times do not depend on the layer (UNI_X).
template <typename T, int NB>
__device__ __forceinline__ void fill_transfers(const BoundSmem &sm, const SProf<T> &sp, int S, int m, int n_seg) {
    const float x0 = __double2float_rd((double)sp.XT[0][0]), x1 = __double2float_rd((double)sp.XT[1][0]);
    for (int s = threadIdx.x; s < n_seg; s += kBoundThreads) {
        const uint64_t tier = sm.segs[s].tier;
        float X = 0.0f;
        int n = 0;
#pragma unroll 4
        for (int i = 4 * NB - 1; i >= 0; --i) {
            if (i < S - 1) {
                const bool far = (tier >> i) & 1ull;
                const float X_up = X;
                X = __fadd_rd(X, 2.0f * (far ? x1 : x0));
                if (far && sp.sched != CM_SCHED_GPIPE) {
                    if (n < kFarMax)
                        sm.far[s * kFarMax + n] = FarVisit{__fmaf_rd(2.0f * stay_pairs(i, S, m), x1, X),
                                                           __fmaf_rd(2.0f * stay_pairs(i + 1, S, m), x1, X_up), i, 0};
                    n = n < kFarMax ? n + 1 : kFarLong;
                }
            }
            sm.xs[s * 4 * NB + i] = X;
        }
        sm.segs[s].n_far = n;
    }
}

// Bound of the lane's composition in one segment, without the slack (bound_of).  What a segment adds -- the
// transfers of its link tiers -- is prepared once per CTA (UNI_X) or worked out per plan.
template <typename T, int NB, bool UNI_X>
__device__ __forceinline__ float lane_value(const LaneBound<NB> &v, const SProf<T> &sp, int S, int m, int s, const BoundSmem &sm) {
    const SegLite &sg = sm.segs[s];
    float best = v.once, x_all;
    if (UNI_X) {
        const float4 *xr = reinterpret_cast<const float4 *>(sm.xs + s * 4 * NB);
        float other = kNoWalk;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            const float4 x = xr[k];
            const float2 p = add2_rd(v.b[2 * k], make_float2(x.x, x.y)), q = add2_rd(v.b[2 * k + 1], make_float2(x.z, x.w));
            best = max3(best, p.x, p.y);
            other = max3(other, q.x, q.y);
            if (k == 0) x_all = x.x;
        }
        if (sg.n_far <= kFarMax) {
            for (int k = 0; k < sg.n_far; ++k) {
                const FarVisit f = sm.far[s * kFarMax + k];
                const float2 r = add2_rd(sm.cd[f.at * kBoundThreads], make_float2(f.up, f.down));
                best = max3(best, r.x, r.y);
            }
        } else {
            const float x1 = __double2float_rd((double)sp.XT[1][0]);
            const float *xf = sm.xs + s * 4 * NB;
            for (uint64_t t = sg.tier; t; t &= t - 1) {
                const int i = __ffsll((long long)t) - 1;
                const float2 cd = sm.cd[i * kBoundThreads];
                best = fmaxf(best, __fadd_rd(cd.x, __fmaf_rd(2.0f * stay_pairs(i, S, m), x1, xf[i])));
                best = fmaxf(best, __fadd_rd(cd.y, __fmaf_rd(2.0f * stay_pairs(i + 1, S, m), x1, i + 1 < S - 1 ? xf[i + 1] : 0.0f)));
            }
        }
        best = fmaxf(best, other);
    } else {
        float X = 0.0f;
#pragma unroll
        for (int i = 4 * NB - 1; i >= 0; --i) {
            if (i < S) {
                if (i < S - 1) {
                    const bool far = (sg.tier >> i) & 1ull;
                    const float x = __double2float_rd((double)sp.XT[far ? 1 : 0][sm.cut[i * kBoundThreads] - 1]);
                    const float X_up = X;
                    X = __fadd_rd(X, 2.0f * x);
                    if (far && sp.sched != CM_SCHED_GPIPE) {
                        const float2 cd = sm.cd[i * kBoundThreads];
                        best = fmaxf(best, __fadd_rd(cd.x, __fmaf_rd(2.0f * stay_pairs(i, S, m), x, X)));
                        best = fmaxf(best, __fadd_rd(cd.y, __fmaf_rd(2.0f * stay_pairs(i + 1, S, m), x, X_up)));
                    }
                }
                best = fmaxf(best, __fadd_rd(v.get(i), X));
            }
        }
        x_all = X;
    }
    return __fmaf_rd(v.g, sg.coef, __fadd_rd(__fadd_rd(v.u0, x_all), best));
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

// Instantiations of the kernel bodies by stages in fours; a depth in between takes the next one.
constexpr int kBoundNb[] = {4, 9, 16};

}  // namespace cm
