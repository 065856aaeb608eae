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
// A stage that outweighs those above it is busy from its first forward to its last backward, and going to
// the top in the meantime takes less time than staying.  A walk along the whole order of a stage has the
// value U_0 - U_a + m w_a; one that goes to the top with the first micro-batch only, U_0 + (m-1) w_a -
// (S-1-a) f_a (the forwards before the first backward are on the way up), with the last only, the same with
// b_a.  With one layer of twenty times the others (random pipelines of 17 to 36 stages) 95 % of the plans
// miss their bound without these, by 16 % of their time in the mean, and 10 % by 0.5 % with them.
// All-forward-all-backward order: climb once, (m-1) extra forwards at the slowest forward, (m-1)
// extra backwards at the slowest backward; with identical micro-batches that is the longest path.
//
// Plans whose bounds tie are told apart by rounding alone, and there are many (every plan with the
// same slowest stage, under the second order).  For them the bound is made exact (walk_time): the
// recurrence adds one duration at a time, and rounded addition is monotone, so the sum along a
// walk, added up in the walk's order in the recurrence's own arithmetic, is still a lower bound of
// the computed time -- bit for bit, and nearly always equal to it -- at 2 (S + m) additions instead
// of 6 S m operations.
#pragma once

#include "cm_plan_eval.cuh"

namespace cm {

// Relative slack between a bound in double arithmetic and the recurrence's rounded result: a path
// has at most 2 (m + S) <= 8320 additions of one rounding each (2^-53), on either side.
constexpr double kBoundSlack = 1.0 - 1.0 / (1ull << 36);

// A list of the bounded search pass was full: the host repeats the search without bounds, and what is left of
// this one need not run.  Threads of a CTA may each look only in kernels beside which none runs that lists plans (all but
// cm_refine_kernel, whose CTAs list them themselves, and cm_gather_kernel): there all of them see the same.
__device__ __forceinline__ bool lists_full(const BatchDev &bd) { return *(volatile unsigned long long *)(bd.counters + 4) == 0ull; }

// Layer cuts of a plan in a shared-memory column, one byte per stage, a plan per thread:
// edge(i) = first layer of stage i, edge(S) = L.
template <int STRIDE> struct CutColumn {
    uint8_t *col;   // col[i * STRIDE] = upper cut of stage i
    __device__ __forceinline__ int edge(int i) const { return i ? col[(i - 1) * STRIDE] : 0; }
    // Returns false if a stage would be empty.
    __device__ __forceinline__ bool fill(CutWalker w, int S) const {
        bool ok = true;
        int lo = 0;
#pragma unroll 4
        for (int i = 0; i < S; ++i) {
            const int hi = w.next();
            col[i * STRIDE] = (uint8_t)hi;
            ok = ok && hi > lo;
            lo = hi;
        }
        return ok;
    }
};

// The best walk of a plan and its value (synchronisation included), in double arithmetic for either
// cost type; value -1 if the plan does not fit in memory (looked at only where no feasible list
// vouches for it).
enum { kWalkStay = 0, kWalkUp = 1, kWalkDown = 2, kWalkForward = 3, kWalkBackward = 4, kWalkAfab = 5, kWalkBusy = 6, kWalkFirst = 7, kWalkLast = 8 };
struct Walk {
    double value;
    long long g_max;    // largest gradient bytes of a stage
    int a, kind, d;     // stage it stays at; what it does there; (kWalkAfab: the stage of the backwards)
};

template <typename T, typename Cuts>
__device__ __forceinline__ Walk best_walk(const SProf<T> &s, const Cuts &c, int S, int m, uint64_t tier, int n_sync, bool check) {
    const bool gpipe = s.sched == CM_SCHED_GPIPE, busy = s.heavy_stage(S);
    double U = 0.0, best = -1.0, fmax = -1.0, bmax = -1.0;
    double base_n = 0.0, w_n = 0.0, q_n = 0.0;   // stage i+1: the value of its own walk (without U_0), w, pairs of stays
    int a = 0, kind = kWalkForward, fa = 0, ba = 0;
    long long g_max = 0;
    int hi = s.L;
    auto take = [&](double v, int at, int k) { if (v > best) { best = v; a = at; kind = k; } };
#pragma unroll 2
    for (int i = S - 1; i >= 0; --i) {
        const int lo = c.edge(i);
        if (check && (hi <= lo || !stage_fits(s.PS[hi] - s.PS[lo], s.PA[hi] - s.PA[lo], i, S, m, s.cap, s.sched)))
            return Walk{-1.0, 0, 0, 0, 0};
        const double f = (double)(s.PF[hi] - s.PF[lo]), bk = (double)(s.PB[hi] - s.PB[lo]), wi = f + bk;
        const double x = i < S - 1 ? 2.0 * (double)s.XT[(tier >> i) & 1ull][hi - 1] : 0.0;
        const long long g = s.PP[hi] - s.PP[lo];
        g_max = g > g_max ? g : g_max;
        if (f > fmax) { fmax = f; fa = i; }
        if (bk > bmax) { bmax = bk; ba = i; }
        U += wi + x;
        if (!gpipe) {
            const int n = m - 1 + i - S;
            const double base = U + (double)n * wi, q = n > 1 ? (double)(n >> 1) : 0.0;
            if (n >= 0) take(base, i, kWalkStay);
            if (i < S - 1) {
                if (q_n > 0.0) take(base_n + q_n * (wi - w_n + x), i + 1, kWalkDown);
                if (q > 0.0) take(base + q * (w_n - wi + x), i, kWalkUp);
            }
            base_n = base; w_n = wi; q_n = q;
            if (busy) {   // uniform
                take((double)m * wi - U, i, kWalkBusy);
                if (n >= -1) take((double)(m - 1) * wi - (double)(S - 1 - i) * (f < bk ? f : bk), i, f < bk ? kWalkFirst : kWalkLast);
            }
        }
        hi = lo;
    }
    if (gpipe) {
        best = (double)(m - 1) * (fmax + bmax);
        a = fa;
        kind = kWalkAfab;
    } else {
        take((double)(m - 1) * fmax, fa, kWalkForward);
        take((double)(m - 1) * bmax, ba, kWalkBackward);
    }
    const double sync = n_sync <= 1 ? 0.0 : (2.0 * (double)(n_sync - 1)) * (double)g_max / ((double)n_sync * (double)s.bw_sync);
    double lb = (U + best + sync) * kBoundSlack;
    if (std::is_same<T, long long>::value || s.intval) lb -= 1.0;   // the quotient floors
    return Walk{lb > 0.0 ? lb : 0.0, g_max, a, kind, ba};
}

// The exact cost along a walk (walk_cost) is at most `goal` for certain: a walk's value is the same sum in double
// arithmetic, less kBoundSlack and one for quotients that floor, and either is rounded at most 2 (m + S) <= 8320 times.
__device__ __forceinline__ bool walk_surely_within(double value, double goal) { return value + 1.0 <= goal * (1.0 - 1.0 / (1ull << 34)); }

// Cost along the walk in the arithmetic and the order of the recurrence: a lower bound of the plan's
// computed cost, bit for bit.
template <typename T, typename Cuts>
__device__ __forceinline__ T walk_cost(const SProf<T> &s, const Cuts &c, int S, int m, uint64_t tier, int n_sync, const Walk &w) {
    T t = (T)0;
    // forwards of stages from .. to-1, each with the transfer above it; backwards of stages from .. to,
    // each with the transfer above it first.  (The additions are one dependent chain; the loads are not.)
    auto climb = [&](int from, int to) {
        int lo = c.edge(from);
#pragma unroll 4
        for (int i = from; i < to; ++i) {
            const int hi = c.edge(i + 1);
            t = t + (s.PF[hi] - s.PF[lo]);
            if (i < S - 1) t = t + s.XT[(tier >> i) & 1ull][hi - 1];
            lo = hi;
        }
    };
    auto drop = [&](int from, int to) {
        int hi = c.edge(from + 1);
#pragma unroll 4
        for (int i = from; i >= to; --i) {
            const int lo = c.edge(i);
            if (i < S - 1) t = t + s.XT[(tier >> i) & 1ull][hi - 1];
            t = t + (s.PB[hi] - s.PB[lo]);
            hi = lo;
        }
    };
    const int a = w.a, lo = c.edge(a), hi = c.edge(a + 1);
    const T f = s.PF[hi] - s.PF[lo], bk = s.PB[hi] - s.PB[lo];
    if (w.kind <= kWalkDown) {
        climb(0, S);
        drop(S - 1, a);
        int n = m - 1 + a - S;
        if (w.kind == kWalkUp) {
            const int hi2 = c.edge(a + 2);
            const T f2 = s.PF[hi2] - s.PF[hi], b2 = s.PB[hi2] - s.PB[hi], x = s.XT[(tier >> a) & 1ull][hi - 1];
            for (; n > 1; n -= 2) t = ((((((t + f) + x) + f2) + b2) + x) + bk);
        } else if (w.kind == kWalkDown) {
            const int lo2 = c.edge(a - 1);
            const T f2 = s.PF[lo] - s.PF[lo2], b2 = s.PB[lo] - s.PB[lo2], x = s.XT[(tier >> (a - 1)) & 1ull][lo - 1];
            for (; n > 1; n -= 2) t = ((((((t + x) + b2) + f2) + x) + f) + bk);
        }
        for (; n > 0; --n) t = (t + f) + bk;
        climb(a, S);
        drop(S - 1, 0);
    } else if (w.kind >= kWalkBusy) {
        const int warm = S - 1 - a < m ? S - 1 - a : m;   // forwards of the stage before its first backward's pair
        climb(0, w.kind == kWalkFirst ? S : a);
        if (w.kind == kWalkFirst) drop(S - 1, a);
        else
            for (int k = warm; k > 0; --k) t = t + f;
        for (int k = w.kind == kWalkBusy ? m - warm : m - 1 - warm; k > 0; --k) t = (t + f) + bk;
        if (w.kind == kWalkLast) {
            climb(a, S);
            drop(S - 1, 0);
        } else {
            for (int k = warm; k > 0; --k) t = t + bk;
            if (a > 0) drop(a - 1, 0);
        }
    } else {
        const bool forwards = w.kind != kWalkBackward, backwards = w.kind != kWalkForward;
        climb(0, a);
        for (int k = forwards ? m - 1 : 0; k > 0; --k) t = t + f;
        climb(a, S);
        const int d = w.kind == kWalkAfab ? w.d : a, dlo = c.edge(d), dhi = c.edge(d + 1);
        const T db = s.PB[dhi] - s.PB[dlo];
        drop(S - 1, d);
        for (int k = backwards ? m - 1 : 0; k > 0; --k) t = t + db;
        if (d > 0) drop(d - 1, 0);
    }
    return t + Num<T>::sync(w.g_max, n_sync, s.bw_sync, s.intval);
}

}  // namespace cm
