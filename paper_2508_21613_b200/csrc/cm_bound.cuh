// Lower bound on the time of one pipeline-plan in O(stages).
//
// The start/end transition equation (Section "Estimator") takes maxima of sums, so the computed
// pipeline time is the largest value of any dependency path; the value of ONE path is a lower
// bound.  In the round order of the 1F1B recurrence (cm_plan_eval.cuh) a path is a walk over
// stages with one step per round t = 0 .. S-2+m: from stage s it moves up to s+1 (forward f_s and
// the transfer x_s) or runs forward and backward at s and may then drop to any lower stage within
// the round (a transfer and a backward per stage).  With w_s = f_s + b_s and
// U_a = sum_{s>=a} w_s + 2 sum_{a<=s<S-1} x_s the walk
//     climb to the top with the first micro-batch (rounds 0 .. S-1), drop to stage a, stay there
//     for rounds S .. m-2+a, climb to the top again with the last micro-batch, drop to stage 0
// has the value U_0 + U_a + (m-1+a-S) w_a (it exists where m-1+a-S >= 0).  Two consecutive stays
// at a may be replaced by a visit to a neighbour, which is worth w_{a+-1} - w_a + 2 x more: the
// bound is the best of the three over all a.  On layer times with a few per cent of spread this
// meets the recurrence to rounding for nearly every plan (mean gap on the 96-layer job below 0.1
// per mille, against 2-3 per cent for the slowest stage alone).  Where m is too small for a
// stage's walk, climbing once and repeating one stage's forwards or backwards,
// U_0 + (m-1) max(f, b), still exists.
// All-forward-all-backward order: climb once, (m-1) extra forwards at the slowest forward, (m-1)
// extra backwards at the slowest backward.
#pragma once

#include "cm_plan_eval.cuh"

namespace cm {

// Relative slack between a bound in double arithmetic and the recurrence's rounded result: a path
// has at most 2 (m + S) <= 8320 additions of one rounding each (2^-53), on either side.
constexpr double kBoundSlack = 1.0 - 1.0 / (1ull << 36);

// Layer cuts of a plan from the last stage to the first.
struct BackWalker {
    uint64_t a, b;
    const uint8_t *row;
    int kind, q, hi;
    __device__ __forceinline__ int lower(int i) {   // lower cut of stage i, for i = S-1, S-2, .., 0
        if (kind == 0) {
            hi -= q + (int)((a >> i) & 1ull);
        } else if (kind == 1) {
            if (i == 0) hi = 0;
            else if (b) { const int v = 63 - __clzll((long long)b); b &= ~(1ull << v); hi = 64 + v + 1; }
            else { const int v = 63 - __clzll((long long)a); a &= ~(1ull << v); hi = v + 1; }
        } else {
            hi = row[i];
        }
        return hi;
    }
};

__device__ __forceinline__ bool make_back_walker(BackWalker &w, const Tables &tb, int layer_mode, int L, int S,
                                                 uint64_t kappa, uint64_t K, uint32_t mm_slot) {
    CutWalker c;
    const bool ok = make_walker(c, tb, layer_mode, L, S, kappa, K, mm_slot);
    w.a = c.a; w.b = c.b; w.row = c.row; w.kind = c.kind; w.q = c.q; w.hi = L;
    return ok;
}

// Bound on the cost (synchronisation included) of one plan of one segment, in double arithmetic for
// either cost type; -1 if the plan does not fit in memory (looked at only where no feasible list
// vouches for it).
template <typename T>
__device__ __forceinline__ double plan_bound(const SProf<T> &s, BackWalker w, int S, int m, uint64_t tier, int n_sync, bool check) {
    const bool gpipe = s.sched == CM_SCHED_GPIPE;
    double U = 0.0, best = 0.0, fmax = 0.0, bmax = 0.0;
    double base_n = 0.0, w_n = 0.0, q_n = 0.0;   // stage i+1: the value of its own walk (without U_0), w, pairs of stays
    long long g_max = 0;
    int hi = s.L;
    for (int i = S - 1; i >= 0; --i) {
        const int lo = w.lower(i);
        if (check && (hi <= lo || !stage_fits(s.PS[hi] - s.PS[lo], s.PA[hi] - s.PA[lo], i, S, m, s.cap, s.sched))) return -1.0;
        const double f = (double)(s.PF[hi] - s.PF[lo]), bk = (double)(s.PB[hi] - s.PB[lo]), wi = f + bk;
        const double x = i < S - 1 ? 2.0 * (double)s.XT[(tier >> i) & 1ull][hi - 1] : 0.0;
        const long long g = s.PP[hi] - s.PP[lo];
        g_max = g > g_max ? g : g_max;
        fmax = tmax(fmax, f);
        bmax = tmax(bmax, bk);
        U += wi + x;
        if (!gpipe) {
            const int n = m - 1 + i - S;
            const double base = U + (double)n * wi, q = n > 1 ? (double)(n >> 1) : 0.0;
            if (n >= 0) best = tmax(best, base);
            if (i < S - 1) {
                if (q_n > 0.0) best = tmax(best, base_n + q_n * (wi - w_n + x));   // stays at i+1, visits to i
                if (q > 0.0) best = tmax(best, base + q * (w_n - wi + x));         // stays at i, visits to i+1
            }
            base_n = base; w_n = wi; q_n = q;
        }
        hi = lo;
    }
    best = tmax(best, (double)(m - 1) * (gpipe ? fmax + bmax : tmax(fmax, bmax)));
    const double sync = n_sync <= 1 ? 0.0 : (2.0 * (double)(n_sync - 1)) * (double)g_max / ((double)n_sync * (double)s.bw_sync);
    double lb = (U + best + sync) * kBoundSlack;
    if (std::is_same<T, long long>::value || s.intval) lb -= 1.0;   // the quotient floors
    return lb > 0.0 ? lb : 0.0;
}

}  // namespace cm
