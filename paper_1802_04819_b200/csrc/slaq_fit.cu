// Normalisation and curve fit.
//
// For every active job: stage the window of stored losses in shared memory, find the largest
// one-step reduction seen so far and scale the window by it ("Normalizing Quality Metrics"),
// then fit both convergence families of "Predicting Quality Improvement",
//     I : f(x) = 1 / (a x^2 + b x + c) + d          II : f(x) = exp(alpha - beta x) + c,
// by exponentially weighted least squares with Levenberg-Marquardt, in window coordinates
// (newest point x = 0, oldest x = -1); the family with the lower weighted residual wins.
//
// Work split.  Jobs are sorted by window length (counting sort, longest first) and cut into
// length classes.  In class c a group of L lanes (L = 2, 4, .. 32: the fewest lanes at which
// the window fits the rows of a warp's shared-memory slice) owns one job (so a warp carries
// 32/L jobs; with fewer jobs L is raised where a shorter chain of rows is worth the work, see
// fit_plan).  One persistent launch (one block of 8, 12 or 16 warps per SM, see fit_plan) serves all classes from one work queue,
// longest windows first.  A lane walks its job's points m = l, l + L, l + 2L, ... counted
// from the newest one; both families
// are evaluated in the same sweep over the window; the partial sums of the normal equations
// are reduced over the L lanes with shuffles; the even lanes of a group then run family I's
// solver step for the job and the odd lanes family II's.  All per-job control flow is per
// lane, so the jobs of a warp may be in different phases of the solver.
// Clusters with fewer jobs than the GPU has sub-partitions take a block per job instead (fit_team_kernel).
#include <math_constants.h>

#include <algorithm>
#include <cmath>

#include "slaq_internal.cuh"
#include "slaq_fit_sweep.cuh"
#include "slaq_log.cuh"

namespace slaq {

namespace {

// Phase clocks (only in a library built with -DSLAQ_PHASE_CLOCKS): lane 0 of every warp adds up the
// SM cycles it spends in each phase of the fit; the totals go to counters[8..13].
struct Phases {
#ifdef SLAQ_PHASE_CLOCKS
    long long sum[6], since;
#endif
};
#ifdef SLAQ_PHASE_CLOCKS
#define SLAQ_PHASE(i)                        \
    do {                                     \
        const long long now_ = clock64();    \
        phases.sum[i] += now_ - phases.since; \
        phases.since = now_;                 \
    } while (0)
#define SLAQ_PHASES_START(p) (p).since = clock64()
#else
#define SLAQ_PHASE(i)
#define SLAQ_PHASES_START(p)
#endif

constexpr int kMaxWarpsPerBlock = 16;          // one block per SM: its warps share one copy of the weight table
constexpr int kTeamWarps = 8;               // warps of a block that works on one job
constexpr size_t kTeamSmem = 220 * 1024;
constexpr double kLambda0 = 1e-3, kLambdaMin = 1e-5, kLambdaMax = 1e12;

// Reductions over the L lanes of a group (L a power of two); every lane of the warp takes part.
__device__ __forceinline__ double group_sum(double v, int L) {
    for (int o = L >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ double group_max(double v, int L) {
    for (int o = L >> 1; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ double group_min(double v, int L) {
    for (int o = L >> 1; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ int group_and(int v, int L) {
    for (int o = L >> 1; o > 0; o >>= 1) v &= __shfl_xor_sync(kFull, v, o);
    return v;
}
__device__ __forceinline__ int warp_max_int(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
    return v;
}

// One asynchronous copy of a double from global to shared memory (both 8-byte aligned).
__device__ __forceinline__ void copy_async_8(double* dst_shared, const double* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_shared);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}

// Copy the job's window into the lane columns (ring storage: the newest loss sits just before
// `head`).  Returns H, or 0 after flagging storage that cannot be right.
template <class Lanes>
__device__ int stage_window(const JobArrays& job, int j, int h_cap, const Lanes& S, int32_t* err_word) {
    if (j < 0) return 0;
    const double* row = job.row[j];
    const int cap = job.cap[j];
    const int H = job.count[j];
    if (H <= 0) return 0;
    if (H > cap || H > h_cap || row == nullptr) {   // never expected: record and skip the job
        if (S.l == 0) atomicOr(err_word, kErrWindow);
        return 0;
    }
#ifdef SLAQ_DEBUG_BOUNDS
    {   // the ring lies inside one of the pools, and the write position inside the ring
        const bool in_ring = row >= job.ring_lo && row + cap <= job.ring_hi;
        const bool in_packed = job.packed_lo && row >= job.packed_lo && row + cap <= job.packed_hi;
        const int head = job.head[j];
        if (!(in_ring || in_packed) || head < 0 || head >= cap) {
            if (S.l == 0) atomicOr(err_word, kErrStorage);
            return 0;
        }
    }
#endif
    int newest = job.head[j] - 1;
    if (newest < 0) newest += cap;
    // asynchronous 8-byte copies straight into the lane's column: all of a lane's points are in
    // flight at once, and nothing passes through registers
    double* dst = S.y + S.lane;
    for (int m = S.l; m < H; m += S.L(), dst += 32) {
        int pos = newest - m;
        pos += pos < 0 ? cap : 0;
        if (index_ok(pos, cap, kErrStorage, err_word) && S.holds(dst)) copy_async_8(dst, row + pos);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    return H;
}

struct Normalised {
    double M;        // largest reduction seen so far
    int status;      // SLAQ_JOB_FITTED here means "usable": M > 0 and everything finite
    double rho;      // weighted mean normalised reduction per iteration (linear extrapolation)
    double ymin, ymax;   // with kRange only
};

// Largest reduction over the window joined with what was seen before it; weighted mean
// normalised change; then the window is scaled in place to levels y = l / M.  k_all: uniform
// trip count of the warp.  changes_out (optional, global, indexed oldest first) receives the
// normalised changes.
//
// A level is l / M correctly rounded.  Where all magnitudes lie between 2^-400 and 2^400 it is formed from the correctly rounded r = 1 / M
// by q = l r, q += (l - q M) r twice: the first correction brings q to within an ulp, the second rounds correctly (Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990), five operations and no test for special cases per row (fit of 100,000 windows of up to 1,000: 3,483 -> 3,448 us; warm started, without the range as well, 1,354 -> 1,307).
// kRange: the lowest and the highest level are wanted (first guesses).
template <bool kRange, class Lanes>
__device__ Normalised normalise_window(const Lanes& S, int H, int k_all, double m_seen, int min_fit_points,
                                       double* changes_out) {
    Normalised out;
    out.M = CUDART_NAN;
    out.rho = 0.0;
    // Rows of the lane with a point (m < H), and with a point that has an older neighbour (m + 1 < H).  The rows
    // that every lane of the warp has are walked without a test per row (a branch in these loops costs issue
    // slots on every row), the ragged rest with one.
    const int shift = __ffs(S.L()) - 1;
    const int rows = H - 1 - S.l >= 0 ? ((H - 1 - S.l) >> shift) + 1 : 0;
    const int rows_nb = H - 2 - S.l >= 0 ? ((H - 2 - S.l) >> shift) + 1 : 0;
    const int full_nb = __reduce_min_sync(kFull, rows_nb);
    const int nb_off = S.l + 1 < S.L() ? 1 : 32 - (S.L() - 1);   // from a point to its older neighbour
    // Largest magnitude, by its high word: 0x7ff00000 and above is not finite.  The running extremes here and below are a compare and
    // a select; fmin and fmax would also sort out NaN (two instructions more per row), which only a window that is
    // refused for it can bring.  These passes are bound by issue (100,000 windows of up to 1,000, with the sign test of
    // first_guesses: fit 3,711 -> 3,615 us, warm started 1,486 -> 1,428).
    int top = 0, bottom = 0x7fffffff;
    double dmax = -CUDART_INF;
    auto magnitude = [&](double v) {
        const int h = __double2hiint(v) & 0x7fffffff;
        top = max(top, h);
        bottom = min(bottom, h);
    };
    auto difference = [&](double older, double v) {
        const double d = older - v;
        if (d > dmax) dmax = d;
    };
    {
        const double* yp = S.y + S.lane;
        int k = 0;
#pragma unroll 2
        for (; k < full_nb; ++k, yp += 32) {
            const double v = S.holds(yp) ? *yp : 0.0;
            magnitude(v);
            difference(S.holds(yp + nb_off) ? yp[nb_off] : 0.0, v);
        }
        for (; k < k_all; ++k, yp += 32) {
            if (k < rows) {
                const double v = S.holds(yp) ? *yp : 0.0;
                magnitude(v);
                if (k < rows_nb) difference(S.holds(yp + nb_off) ? yp[nb_off] : 0.0, v);
            }
        }
    }
    const int fin = group_and(top < 0x7ff00000 ? 1 : 0, S.L());
    dmax = group_max(dmax, S.L());
    if (H <= 0) {
        out.status = SLAQ_JOB_INACTIVE;
    } else if (!fin || m_seen != m_seen || m_seen == CUDART_INF) {
        out.status = SLAQ_JOB_NONFINITE;
    } else if (H == 1) {
        out.status = SLAQ_JOB_NEW;
    } else {
        out.M = fmax(m_seen, dmax);
        out.status = (out.M > 0.0 && finite_d(out.M)) ? SLAQ_JOB_FITTED : SLAQ_JOB_FLAT;
    }
    const bool usable = out.status == SLAQ_JOB_FITTED;
    const double M = out.M;
    // the normalised changes feed only the linear extrapolation of short windows (and the export)
    const bool want_changes = usable && (H < min_fit_points || changes_out != nullptr);
    double num = 0.0, den = 0.0;
    if (__any_sync(kFull, want_changes)) {
        for (int k = 0; k < k_all; ++k) {
            const int m = S.l + S.L() * k;
            if (want_changes && m + 1 < H) {
                const double change = __ddiv_rn(older_neighbour(S, k) - S.level(k), M);
                const double w = S.weight(m);
                num = fma(w, change, num);
                den += w;
                if (changes_out) changes_out[H - 1 - m] = change;
            }
        }
        if (changes_out && usable && S.l == 0) changes_out[0] = 0.0;
        num = group_sum(num, S.L());
        den = group_sum(den, S.L());
        out.rho = fmax(num / den, 0.0);
    }
    __syncwarp();   // all neighbour reads are done before the window is overwritten
    double lo = CUDART_INF, hi = -CUDART_INF;
    // unusable jobs keep their window as it is: they count as lanes without rows
    const int own = usable ? rows : 0;
    const int full = __reduce_min_sync(kFull, own);
    auto scale = [&](auto level) {
        auto one = [&](double* yp) {
            const double y = level(S.holds(yp) ? *yp : 0.0);
            if (S.holds(yp)) *yp = y;
            if (kRange) {
                if (y < lo) lo = y;
                if (y > hi) hi = y;
            }
        };
        double* yp = S.y + S.lane;
        int k = 0;
#pragma unroll 2
        for (; k < full; ++k, yp += 32) one(yp);
        for (; k < k_all; ++k, yp += 32)
            if (k < own) one(yp);
    };
    constexpr int kLeast = (1023 - 400) << 20, kMost = (1023 + 400) << 20;   // high words
    const int hM = __double2hiint(M);
    const bool plain = own == 0 || (bottom >= kLeast && top < kMost && hM >= kLeast && hM < kMost);
    if (__all_sync(kFull, plain)) {
        const double r = __drcp_rn(M);
        scale([&](double v) {
            double q = v * r;
            q = fma(fma(-q, M, v), r, q);
            return fma(fma(-q, M, v), r, q);
        });
    } else {
        scale([&](double v) { return __ddiv_rn(v, M); });
    }
    if (kRange) {
        out.ymin = group_min(lo, S.L());
        out.ymax = group_max(hi, S.L());
    }
    __syncwarp();
    return out;
}

// The lowest and the highest level of the scaled window, where normalise_window did not look for them.
template <class Lanes>
__device__ void level_range(const Lanes& S, int H, int k_all, Normalised& nz) {
    double lo = CUDART_INF, hi = -CUDART_INF;
    for (int k = 0; k < k_all; ++k) {
        if (S.l + S.L() * k < H) {
            const double y = S.level(k);
            if (y < lo) lo = y;
            if (y > hi) hi = y;
        }
    }
    nz.ymin = group_min(lo, S.L());
    nz.ymax = group_max(hi, S.L());
}

// Weighted mean normalised change per iteration from the scaled window (used when a window long
// enough for a fit ends without one): sum w (y_{i-1} - y_i) / sum w.
template <class Lanes>
__device__ double mean_change_of_levels(const Lanes& S, int H, int k_all) {
    double num = 0.0, den = 0.0;
    for (int k = 0; k < k_all; ++k) {
        const int m = S.l + S.L() * k;
        if (m + 1 < H) {
            const double w = S.weight(m);
            num = fma(w, older_neighbour(S, k) - S.level(k), num);
            den += w;
        }
    }
    num = group_sum(num, S.L());
    den = group_sum(den, S.L());
    return fmax(num / den, 0.0);
}

// ---- small dense algebra: every lane solves its own job's system ----

struct Sym4 {   // symmetric 4x4, upper triangle
    double a00, a01, a02, a03, a11, a12, a13, a22, a23, a33;
};

// Solve B x = r for symmetric positive definite B by the root-free Cholesky factorisation
// B = L D L^T.  False if a pivot is not positive and finite or the solution is not finite.  Unknowns whose bit is set
// in `fixed` (of the first three) are left out and come back as 0: a pivot's reciprocal taken as 0 removes its row and
// column.
__device__ bool ldl_solve(const Sym4& B, const double (&r)[4], unsigned fixed, double (&x)[4]) {
    const bool f0 = fixed & 1u, f1 = fixed & 2u, f2 = fixed & 4u;
    const double d0 = B.a00;
    const double i0 = f0 ? 0.0 : fast_rcp(d0);
    const double l10 = B.a01 * i0, l20 = B.a02 * i0, l30 = B.a03 * i0;
    const double d1 = fma(-l10, B.a01, B.a11);
    const double i1 = f1 ? 0.0 : fast_rcp(d1);
    const double t21 = fma(-l20, B.a01, B.a12), t31 = fma(-l30, B.a01, B.a13);
    const double l21 = t21 * i1, l31 = t31 * i1;
    const double d2 = fma(-l21, t21, fma(-l20, B.a02, B.a22));
    const double i2 = f2 ? 0.0 : fast_rcp(d2);
    const double t32 = fma(-l31, t21, fma(-l30, B.a02, B.a23));
    const double l32 = t32 * i2;
    const double d3 = fma(-l32, t32, fma(-l31, t31, fma(-l30, B.a03, B.a33)));
    const double i3 = fast_rcp(d3);
    // positive and finite, read off the high words (a subnormal pivot counts as zero: its reciprocal is not finite)
    const int fine = 0x3ff00000;
    const int h0 = f0 ? fine : __double2hiint(d0), h1 = f1 ? fine : __double2hiint(d1), h2 = f2 ? fine : __double2hiint(d2);
    const int h3 = __double2hiint(d3);
    bool ok = min(min(h0, h1), min(h2, h3)) > 0 && max(max(h0, h1), max(h2, h3)) < 0x7ff00000;
    const double z0 = r[0];
    const double z1 = fma(-l10, z0, r[1]);
    const double z2 = fma(-l21, z1, fma(-l20, z0, r[2]));
    const double z3 = fma(-l32, z2, fma(-l31, z1, fma(-l30, z0, r[3])));
    x[3] = z3 * i3;
    x[2] = fma(-l32, x[3], z2 * i2);
    x[1] = fma(-l31, x[3], fma(-l21, x[2], z1 * i1));
    x[0] = fma(-l30, x[3], fma(-l20, x[2], fma(-l10, x[1], z0 * i0)));
    const int m = 0x7ff00000;
    ok = ok && max(max(__double2hiint(x[0]) & m, __double2hiint(x[1]) & m),
                   max(__double2hiint(x[2]) & m, __double2hiint(x[3]) & m)) < m;
    return ok;
}

// Solver state of ONE family for one job.  The lanes of a group alternate: even lanes carry
// family I, odd lanes family II, so one instruction stream advances both solvers at once.
struct Family {
    double p[4];       // current parameters
    double S;          // weighted residual at p
    double lambda, nu;
    double inv_predicted;   // one over the reduction the quadratic model promises for the trial step; 0 if it promises none
    unsigned was_frozen;
    int sweeps;
    bool ok;           // the starting point was usable
    bool done;         // no further trials
    bool has_trial;    // the running sweep evaluates the trial point
};

// One Levenberg-Marquardt trial up to the point where the model must be evaluated: freeze
// parameters that sit on their bound while the descent direction or the solved step points
// outside (and keep them frozen from then on), solve (A + lambda diag A) step = g over the
// rest, clip the trial point to the bounds, and record the reduction the quadratic model
// promises.  Lower bounds: a >= 0, b >= 0, c >= 1e-12 of family I keep the curve non-increasing ahead of the newest
// point and its denominator positive there; beta >= 0 of family II.  `busy` = this lane has a trial to prepare; the
// re-solve loop runs while any lane of the warp needs another round (each freezes at least one more of the three
// bounded parameters).  Family II has three parameters: the fourth row of its system is empty but for the diagonal.
// kRows, rows: x counts rows, and the window's length in that unit.
template <bool kRows>
__device__ void prepare_trial(Family& F, int fam, const Sym4& A, const double (&g)[4], bool busy, double tiny_S,
                              double rows, double (&trial)[4]) {
    F.has_trial = false;
    if (busy && F.S <= tiny_S) {   // residual is zero to rounding
        F.done = true;
        busy = false;
    }
    const bool one = fam == 0;
    // on their bounds; no parameter with bound 0 is ever below it, so the high word tells (subnormals count as 0)
    const bool at0 = one && __double2hiint(F.p[0]) <= 0, at1 = __double2hiint(F.p[1]) <= 0, at2 = one && F.p[2] <= 1e-12;
    unsigned frozen = 0;
    if (at0 && (__double2hiint(g[0]) < 0 || (F.was_frozen & 1u))) frozen |= 1u;
    if (at1 && (__double2hiint(g[1]) < 0 || (F.was_frozen & 2u))) frozen |= 2u;
    if (at2 && (__double2hiint(g[2]) < 0 || (F.was_frozen & 4u))) frozen |= 4u;
    // The damped diagonal.  An entry below 1e-300 in the window's unit (a curve that has run off to infinity everywhere but at the
    // newest point) is damped by that.
    Sym4 B = A;
    if constexpr (kRows) {
        B.a00 = fma(F.lambda, A.a00, A.a00), B.a11 = fma(F.lambda, A.a11, A.a11);
        B.a22 = fma(F.lambda, A.a22, A.a22), B.a33 = fma(F.lambda, A.a33, A.a33);
        // 0x05000000 is the high word of some 1e-285, above 1e-300 in any unit
        if (min(min(__double2hiint(A.a00), __double2hiint(A.a11)), min(__double2hiint(A.a22), __double2hiint(A.a33))) < 0x05000000) {
            const double f = rows * rows;   // a power of x on either side of the product makes it rows times the window's value
            auto damped = [&](double d, double least) { return fma(F.lambda, d < least ? least : d, d); };
            B.a00 = damped(A.a00, one ? 1e-300 * f * f : 1e-300), B.a11 = damped(A.a11, 1e-300 * f);
            B.a22 = damped(A.a22, 1e-300), B.a33 = damped(A.a33, 1e-300);
        }
    } else {   // 0x01a56e1f is the high word of 1e-300
        auto damped = [&](double d) { return fma(F.lambda, __double2hiint(d) < 0x01a56e1f ? 1e-300 : d, d); };
        B.a00 = damped(A.a00), B.a11 = damped(A.a11), B.a22 = damped(A.a22), B.a33 = damped(A.a33);
    }
    double step[4] = {0.0, 0.0, 0.0, 0.0};
    bool solved = false, again = busy;
    while (__any_sync(kFull, again)) {
        if (again) {
            solved = ldl_solve(B, g, frozen, step);
            unsigned grow = 0;
            if (at0 && __double2hiint(step[0]) < 0) grow |= 1u;
            if (at1 && __double2hiint(step[1]) < 0) grow |= 2u;
            if (at2 && __double2hiint(step[2]) < 0) grow |= 4u;
            grow = solved ? grow & ~frozen : 0u;
            frozen |= grow;
            again = grow != 0;
        }
    }
    if (!busy) return;
    F.was_frozen |= frozen;
    if (!solved) {   // no step: counts as a rejected trial
        F.lambda = fmin(F.lambda * F.nu, kLambdaMax);
        F.nu *= 2.0;
        return;
    }
    double d[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) trial[a] = F.p[a] + step[a];
    if (one && __double2hiint(trial[0]) < 0) trial[0] = 0.0;
    if (__double2hiint(trial[1]) < 0) trial[1] = 0.0;
    if (one && trial[2] < 1e-12) trial[2] = 1e-12;
#pragma unroll
    for (int a = 0; a < 4; ++a) d[a] = trial[a] - F.p[a];
    const double dg = fma(d[0], g[0], fma(d[1], g[1], fma(d[2], g[2], d[3] * g[3])));
    const double Ad0 = fma(A.a00, d[0], fma(A.a01, d[1], fma(A.a02, d[2], A.a03 * d[3])));
    const double Ad1 = fma(A.a01, d[0], fma(A.a11, d[1], fma(A.a12, d[2], A.a13 * d[3])));
    const double Ad2 = fma(A.a02, d[0], fma(A.a12, d[1], fma(A.a22, d[2], A.a23 * d[3])));
    const double Ad3 = fma(A.a03, d[0], fma(A.a13, d[1], fma(A.a23, d[2], A.a33 * d[3])));
    const double dAd = fma(d[0], Ad0, fma(d[1], Ad1, fma(d[2], Ad2, d[3] * Ad3)));
    // inverted here, where nothing waits for it, and not between the sweep and the next step
    const double predicted = 2.0 * dg - dAd;
    F.inv_predicted = predicted > 0.0 ? fast_rcp(predicted) : 0.0;
    F.has_trial = true;
    F.sweeps += 1;   // every solved trial costs one sweep over the window
}

// After the sweep at the trial point: accept it only if the residual strictly fell, and move
// the damping by the gain ratio (Madsen, Nielsen, Tingleff 2004).  Returns whether accepted.
__device__ __forceinline__ bool finish_trial(Family& F, const double (&trial)[4], bool ok_trial, double S_trial) {
    if (!F.has_trial) return false;
    F.has_trial = false;
    if (ok_trial && S_trial < F.S) {
        const double S_before = F.S;
#pragma unroll
        for (int a = 0; a < 4; ++a) F.p[a] = trial[a];
        F.S = S_trial;
        const double rho = (S_before - S_trial) * F.inv_predicted;
        const double c = 2.0 * rho - 1.0;
        F.lambda *= fmax(1.0 / 3.0, 1.0 - c * c * c);
        F.nu = 2.0;
        F.lambda = fmin(fmax(F.lambda, kLambdaMin), kLambdaMax);
        if (S_before - S_trial <= 1e-14 * S_before) F.done = true;
        return true;
    }
    F.lambda = fmin(F.lambda * F.nu, kLambdaMax);
    F.nu *= 2.0;
    return false;
}

// The sums of the last accepted point live in shared memory between sweeps, one column per job
// and family: every lane writes the ones it holds.  Every lane of the warp calls this; `keep` says
// whether the lane's family has new sums to park.
template <class Lanes>
__device__ __forceinline__ void park(const Lanes& S, const SweepSums& s, bool keep) {
    if (keep) {
        const int n = S.park_stride();
        if (S.L() == 2) {
#pragma unroll
            for (int k = 0; k < kParked; ++k)
                if (S.holds(S.park + k * n)) S.park[k * n] = s.v[k];
        } else {
            int from, own;
            S.held(from, own);
            own = min(own, kParked - from);   // the objective is not parked
            double* const at = S.park + from * n;
            const int most = S.L() == 32 ? 1 : S.L() == 16 ? 2 : S.L() == 8 ? 4 : 7;
#pragma unroll
            for (int k = 0; k < 7; ++k) {
                if (k >= most) break;
                if (k < own && S.holds(at + k * n)) at[k * n] = s.v[k];
            }
        }
    }
    __syncwarp();
}

// Normal equations A = sum w J J^T, g = sum w J r of the lane's family from the parked sums.
template <class Lanes>
__device__ __forceinline__ void normal_equations(const Lanes& S, int fam, double sw, Sym4& A, double (&g)[4]) {
    const double* c = S.park;
    const int n = S.park_stride();
    if (!S.holds(c) || !S.holds(c + (kParked - 1) * n)) {   // bounds build only: leave the system empty
        A = Sym4{0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        g[0] = g[1] = g[2] = g[3] = 0.0;
        return;
    }
    const bool one = fam == 0;
    const double c0 = c[0], c2 = c[2 * n], c5 = c[5 * n];
    A.a00 = c[4 * n]; A.a01 = c[3 * n]; A.a02 = one ? c2 : c5; A.a11 = c2; A.a12 = c[1 * n]; A.a22 = one ? c0 : sw;
    A.a03 = -c[7 * n]; A.a13 = -c[6 * n]; A.a23 = one ? -c5 : 0.0; A.a33 = sw;
    g[0] = -c[10 * n]; g[1] = -c[9 * n]; g[2] = -c[8 * n]; g[3] = c[11 * n];
}

struct Moments {
    double sw, swy2;
};

// First guesses.  d0 lies below every level; with the offset fixed at d0, 1/(y - d0) is a
// quadratic in x (family I: weighted linear least squares, or the line through the oldest and
// newest transformed points if that fit is not a decreasing curve with a positive denominator)
// and log(y - d0) is a line in x (family II: weighted linear regression).  needI / needII: the
// job wants that family's guess (a family that starts from last epoch's parameters does not);
// the weight sums in `mom` are always produced.
// The sums of the weights times powers of x depend on the window's length alone and come from a table: formed in the pass they
// were 7 of its 50 fp64 instructions per point, and 5 of 11 reductions.
struct GuessSums {
    double swy2, r0, r1, r2, su, sxu;
};

// One point of the first-guess pass.  kI / kII: the transformed values of family I (1 / (y - d0)) and of
// family II (log(y - d0)) are wanted by some lane of the warp.  kAny: y - d0 may be subnormal or not finite.
template <bool kI, bool kII, bool kAny, class Lanes>
__device__ __forceinline__ void guess_point(const Lanes& S, const double* wp, const double* yp, double md, double inv_span,
                                            double d0, GuessSums& g) {
    const double x = -md * inv_span;
    const double w = S.weight(wp);
    const double y = S.holds(yp) ? *yp : 0.0;
    g.swy2 = fma(w * y, y, g.swy2);
    if (kI) {
        const double wz = w * fast_rcp(y - d0);
        g.r2 += wz;
        g.r1 = fma(wz, x, g.r1);
        g.r0 = fma(wz * x, x, g.r0);
    }
    if (kII) {
        const double wu = w * (kAny ? log(y - d0) : log_of_normal(y - d0, S.log_table()));
        g.su += wu;
        g.sxu = fma(wu, x, g.sxu);
    }
}

// The rows every lane of the warp has without a test per row, the ragged rest with one.
template <bool kI, bool kII, bool kAny, class Lanes>
__device__ __forceinline__ void guess_rows(const Lanes& S, int own, int k_all, double inv_span, double d0, GuessSums& g) {
    const int full = __reduce_min_sync(kFull, own);
    const double* yp = S.y + S.lane;
    const double* wp = S.wtab + S.l;
    double md = (double)S.l;
    const double dL = (double)S.L();
    int k = 0;
#pragma unroll 1
    for (; k < full; ++k, md += dL, yp += 32, wp += S.L()) guess_point<kI, kII, kAny>(S, wp, yp, md, inv_span, d0, g);
#pragma unroll 1
    for (; k < k_all; ++k, md += dL, yp += 32, wp += S.L())
        if (k < own) guess_point<kI, kII, kAny>(S, wp, yp, md, inv_span, d0, g);
}

template <class Lanes>
__device__ void first_guesses(const Lanes& S, int H, int k_all, double inv_span, double ymin, double ymax, bool busy,
                              bool needI, bool needII, Moments& mom, double (&pI)[4], double (&pII)[4]) {
    constexpr bool kTable = Lanes::kRowUnit;   // log() for teams, where a lane takes one or two, and for warm starts, which take none
    const double d0 = ymax > ymin ? ymin - 0.1 * (ymax - ymin) : ymin - 1e-3 * fmax(fabs(ymin), 1.0);
    GuessSums g = {};
    const int shift = __ffs(S.L()) - 1;
    const int own = busy && H - 1 - S.l >= 0 ? ((H - 1 - S.l) >> shift) + 1 : 0;   // the lane's rows
    // a family that no lane of the warp wants a guess for is left out of the pass; a lane that does not want
    // what the warp computes gets sums it does not use
    const bool anyI = __any_sync(kFull, needI), anyII = __any_sync(kFull, needII);
    // y - d0 lies between its values at the lowest and the highest level (rounding keeps the order)
    const int least = __double2hiint(ymin - d0), most = __double2hiint(ymax - d0);
    const bool odd_one = needII && (least < 0x00100000 || least >= 0x7ff00000 || most < 0x00100000 || most >= 0x7ff00000);
    if (kTable && __any_sync(kFull, odd_one)) {
        guess_rows<true, true, true>(S, own, k_all, inv_span, d0, g);
    } else if (anyI && anyII) {
        guess_rows<true, true, !kTable>(S, own, k_all, inv_span, d0, g);
    } else {
        if (anyI) guess_rows<true, false, !kTable>(S, own, k_all, inv_span, d0, g);
        else if (anyII) guess_rows<false, true, !kTable>(S, own, k_all, inv_span, d0, g);
        else guess_rows<false, false, !kTable>(S, own, k_all, inv_span, d0, g);
    }
    double wm[5];
#pragma unroll
    for (int p = 0; p < 5; ++p) wm[p] = busy && index_ok(H, S.wtab_len + 1, kErrShared, S.err_word) ? S.wsum[p * (S.wtab_len + 1) + H] : 0.0;
    const double inv2 = inv_span * inv_span;
    const double sw = wm[0], swx = -wm[1] * inv_span, swx2 = wm[2] * inv2, swx3 = -wm[3] * (inv2 * inv_span), swx4 = wm[4] * (inv2 * inv2);
    double swy2 = g.swy2;
    double r0 = g.r0, r1 = g.r1, r2 = g.r2, su = g.su, sxu = g.sxu;
    for (int o = S.L() >> 1; o > 0; o >>= 1) {
        swy2 += __shfl_xor_sync(kFull, swy2, o);
        r0 += __shfl_xor_sync(kFull, r0, o); r1 += __shfl_xor_sync(kFull, r1, o);
        r2 += __shfl_xor_sync(kFull, r2, o); su += __shfl_xor_sync(kFull, su, o);
        sxu += __shfl_xor_sync(kFull, sxu, o);
    }
    mom.sw = sw;
    mom.swy2 = swy2;
    // family I
    if (__any_sync(kFull, needI)) {
        Sym4 B;
        B.a00 = swx4; B.a01 = swx3; B.a02 = swx2; B.a11 = swx2; B.a12 = swx; B.a22 = sw;
        B.a03 = B.a13 = B.a23 = 0.0; B.a33 = 1.0;
        const double rhs[4] = {r0, r1, r2, 0.0};
        double sol[4] = {0.0, 0.0, 0.0, 0.0};
        bool good = needI && ldl_solve(B, rhs, 0u, sol) && sol[0] >= 0.0 && sol[1] >= 0.0;
        // Positive at every point?  A curve with a >= 0 is convex, so its lowest value lies at one of the two points on either side
        // of its vertex at m = b / (2 a) span (the oldest point if that lies beyond it, or a = b = 0); a pass over
        // the window's points took a 70th of a cold fit.
        const double m_old_d = (double)(H - 1);
        const double m_left = floor(fmax(fmin(0.5 * sol[1] / (sol[0] * inv_span), m_old_d), 0.0));
        const double x_left = -m_left * inv_span, x_right = -fmin(m_left + 1.0, m_old_d) * inv_span;
        good = good && fma(fma(sol[0], x_left, sol[1]), x_left, sol[2]) > 0.0 && fma(fma(sol[0], x_right, sol[1]), x_right, sol[2]) > 0.0;
        // the oldest point (m = H - 1) and the newest (m = 0), read from the lanes that own them
        const int m_old = max(H - 1, 0);
        const double* at_old = S.y + (m_old / S.L()) * 32 + (S.lane - S.l) + (m_old & (S.L() - 1));
        const double y_old = S.holds(at_old) ? *at_old : 0.0;
        const double y_new = S.holds(S.y + S.lane - S.l) ? S.y[S.lane - S.l] : 0.0;
        if (good) {
            pI[0] = sol[0]; pI[1] = sol[1]; pI[2] = sol[2];
        } else {
            const double z_old = 1.0 / (y_old - d0), z_new = 1.0 / (y_new - d0);
            pI[0] = 0.0;
            pI[1] = fmax(z_new - z_old, 0.0);
            pI[2] = z_new;
        }
        pI[3] = d0;
    }
    // family II
    const double den = sw * swx2 - swx * swx;
    const double slope = (sw * sxu - swx * su) / den;
    pII[0] = (su - slope * swx) / sw;
    pII[1] = fmax(-slope, 1e-8);
    pII[2] = d0;
    pII[3] = 0.0;
}

// Last epoch's end points of both families in this epoch's window coordinates.  The curves
// are functions of the iteration index and the raw loss; with x0 = (k - K0)/span0, y0 = l/M0
// then and x = (k - K)/span, y = l/M now, x0 = t + r x and y = sigma y0, where
// t = (K - K0)/span0, r = span/span0, sigma = M0/M, and both families keep their form under
// that substitution.  Clears `wmask` if the stored coordinates cannot be used.
__device__ void carry_over(const FitArrays& fit, const JobArrays& job, int j, double span, double M, unsigned& wmask,
                           double (&pI)[4], double (&pII)[4]) {
    const double span0 = fit.warm_span[j], M0 = fit.warm_scale[j];
    if (!(span0 > 0.0) || !(M0 > 0.0) || !finite_d(M0)) {
        wmask = 0;
        return;
    }
    const double* q = fit.warm_p + 8 * (size_t)j;
    const double t = (double)(job.k_last[j] - fit.warm_k[j]) / span0;
    const double r = span / span0, sigma = M0 / M;
    if (wmask & 1u) {
        const double a = q[0], b = q[1], c = q[2], d = q[3];
        pI[0] = a * r * r / sigma;
        pI[1] = (2.0 * a * t + b) * r / sigma;
        pI[2] = ((a * t + b) * t + c) / sigma;
        pI[3] = sigma * d;
    }
    if (wmask & 2u) {
        pII[0] = q[4] - q[5] * t + log(sigma);
        pII[1] = q[5] * r;
        pII[2] = sigma * q[6];
        pII[3] = 0.0;
    }
}

// Both families' parameters in another unit of x, f old ones long.  Cold fits count x in rows of a lane's points (x = -m / L): the row
// pitch is then 1, so that x steps exactly, no power of it is multiplied into the sums, and four registers fewer are spilled (100,000
// windows of up to 1,000, with the logarithm by table: 3,615 -> 3,511 us).  The damping scales with the diagonal, so the iteration is the same in every unit.
// Warm starts stay in the window's unit (a curve that ran off to infinity is carried over to a double root at one of the window's points,
// which only the window's unit meets exactly), and so do teams, whose lanes have a row or two.
__device__ __forceinline__ void rescale(double (&pI)[4], double (&pII)[4], double f) {
    pI[0] *= f * f;
    pI[1] *= f;
    pII[1] *= f;
}

// A warm start's first guesses, out of line: most warps of a loop need none, and in line they cost the others registers (944 bytes
// spilled instead of 200; fit of 100,000 windows of up to 1,000: 1,307 against 1,278 us).
template <class Lanes>
__device__ __noinline__ void warm_first_guesses(const Lanes& S, int H, int k_all, double inv_span, bool fits, bool needI, bool needII,
                                                Moments* mom, double* gI, double* gII) {
    Normalised nz;
    level_range(S, H, k_all, nz);
    Moments found;
    double one[4] = {0.0, 0.0, 0.0, 0.0}, two[4] = {0.0, 0.0, 0.0, 0.0};
    first_guesses(S, H, k_all, inv_span, nz.ymin, nz.ymax, fits, needI, needII, found, one, two);
    *mom = found;
#pragma unroll
    for (int a = 0; a < 4; ++a) gI[a] = one[a], gII[a] = two[a];
}

// The sums of first_guesses that do not depend on a guess.
template <class Lanes>
__device__ __forceinline__ void weight_moments(const Lanes& S, int H, int k_all, double inv_span, bool busy, Moments& mom) {
    GuessSums g = {};
    const int shift = __ffs(S.L()) - 1;
    const int own = busy && H - 1 - S.l >= 0 ? ((H - 1 - S.l) >> shift) + 1 : 0;
    guess_rows<false, false, false>(S, own, k_all, inv_span, 0.0, g);
    mom.sw = busy && index_ok(H, S.wtab_len + 1, kErrShared, S.err_word) ? S.wsum[H] : 0.0;
    mom.swy2 = group_sum(g.swy2, S.L());
}

// The second round of a warm start: the families whose carried-over point had no finite
// residual (`redo`, per lane for its own family) take their first guesses and are swept again.
template <class Lanes>
__device__ __noinline__ void restart_from_first_guesses(const Lanes& S, int fam, int H, int k_all, double inv_span,
                                                        double ymin, double ymax, bool fits, bool redo, double* pI,
                                                        double* pII, SweepSums* sums) {
    const int lane = S.lane;
    const bool redoI = __shfl_sync(kFull, (int)redo, lane & ~1) != 0;
    const bool redoII = __shfl_sync(kFull, (int)redo, lane | 1) != 0;
    Moments mom;
    double gI[4], gII[4], qI[4], qII[4];
    first_guesses(S, H, k_all, inv_span, ymin, ymax, fits, redoI, redoII, mom, gI, gII);
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        qI[a] = redoI ? gI[a] : pI[a];
        qII[a] = redoII ? gII[a] : pII[a];
        pI[a] = qI[a];
        pII[a] = qII[a];
    }
    SweepSums again;
    sweep(S, fam, H, k_all, inv_span, qI, redoI, qII, redoII, again);
    if (redo) *sums = again;
}

// One slot of the work queue: the place-th warp's worth of jobs of class c.  kWarm: families may start from last epoch's
// parameters (a separate instantiation, so that the plain one carries none of that code).  kL: lanes per job, a
// constant, which takes branches and index arithmetic out of every step of a trial.
template <bool kWarm, int kL, bool kRows, int kStep, bool kTeam = false>
__device__ __forceinline__ void fit_slot(const JobArrays& job, const FitArrays& fit, const int32_t* __restrict__ order,
                                         const int32_t* __restrict__ start, const FitClasses& cls, int c, int place, int lm_trials,
                                         int min_fit_points, const double* wtab, const double* wsum, double* slice, unsigned long long* tally,
                                         int lane,
                                         Phases& phases, int32_t* err_word, Team team = {}) {
    const int fam = kTeam ? team.fam : lane & 1;   // even lanes solve family I, odd lanes family II
    const bool leader = !kTeam || (team.fam == 0 && team.part == 0);   // writes the job's record
    const int even = lane & ~1, oddl = lane | 1;
    constexpr int L = kL;
    const int h_hi = cls.h_hi[c];
    LanesOf<kL, kRows, kStep> S;
    S.wtab = wtab;
    S.wsum = wsum;
    S.lane = lane;
    S.slice = slice;
    S.slice_len = cls.slice;
    S.wtab_len = cls.h_max;
    S.err_word = err_word;
    S.any_L = L;
    S.l = lane & (L - 1);
    const int G = 32 / L, g = lane / L;
    S.park = slice + 2 * g + (kTeam ? 0 : lane & 1);
    S.y = slice + kParked * 2 * G;
    const int last = order ? start[cls.h_lo[c]] : job.max_jobs;
    const int base = (order ? start[h_hi] : 0) + place * G;
    const int idx = base + g;
    int j = idx < last && index_ok(idx, job.max_jobs, kErrJob, err_word) ? (order ? order[idx] : idx) : -1;
    if (j >= 0 && !index_ok(j, job.max_jobs, kErrJob, err_word)) j = -1;
    __syncwarp();
    const int H = stage_window(job, j, h_hi, S, err_word);
    const int k_all = warp_max_int((H + L - 1) / L);
    __syncwarp();
    const double m_seen = j >= 0 ? job.m_seen[j] : -CUDART_INF;
    Normalised nz = normalise_window<!kWarm>(S, H, k_all, m_seen, min_fit_points, nullptr);
    SLAQ_PHASE(0);   // staging and normalisation

    int status = nz.status, family = -1;
    double p_out[4] = {CUDART_NAN, CUDART_NAN, CUDART_NAN, CUDART_NAN};
    double S_out[2] = {CUDART_INF, CUDART_INF};
    int sweeps_out[2] = {0, 0};
    int ended = 0;   // bit 0 / 1: family I / II ended with a finite residual
    bool any_ended = false;
    double both_out[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // both families' end points
    const double span = (double)max(H - 1, 1);
    const bool fits = status == SLAQ_JOB_FITTED && H >= min_fit_points;   // this lane's job gets curves fitted

    if (__any_sync(kFull, fits)) {
        const double inv_span = 1.0 / span;
        const double pitch = kRows ? (double)L : span;   // points per unit of x
        Moments mom = {0.0, 0.0};
        Family F = {};
        double pI[4] = {0.0, 0.0, 0.0, 0.0}, pII[4] = {0.0, 0.0, 0.0, 0.0};   // the points the next sweep evaluates
        // Starting points: the first guesses, or (kWarm) last epoch's parameters where the job
        // has some; a carried-over point without a finite residual is dropped for the
        // family's first guess in a second round.
        int spent = 0;
        SweepSums sums = {};
        const bool wantsI = fits && (!kTeam || fam == 0), wantsII = fits && (!kTeam || fam == 1);
        auto sweep_at = [&](bool doI, bool doII) {
            if constexpr (kTeam) {
                if (fam == 0) sweep_team<0>(S, team, H, inv_span, pI, sums);
                else sweep_team<1>(S, team, H, inv_span, pII, sums);
            } else {
                sweep(S, fam, H, k_all, inv_span, pI, doI, pII, doII, sums);
            }
        };
        auto park_sums = [&](bool keep) {
            if constexpr (kTeam) {
                if (keep && team.index >= 0 && S.holds(S.park + 2 * team.index)) S.park[2 * team.index] = sums.v[0];
                __syncwarp();
            } else {
                park(S, sums, keep);
            }
        };
        if (!kWarm) {
            first_guesses(S, H, k_all, inv_span, nz.ymin, nz.ymax, fits, wantsI, wantsII, mom, pI, pII);
            if (kRows) rescale(pI, pII, pitch / span);
            sweep_at(fits, fits);
        } else {
            unsigned wmask = fits ? fit.warm_mask[j] : 0u;
            if (wmask) carry_over(fit, job, j, span, nz.M, wmask, pI, pII);
            {
                double gI[4], gII[4];
                const bool needI = wantsI && !(wmask & 1u), needII = wantsII && !(wmask & 2u);
                if (__any_sync(kFull, needI || needII)) {
                    Moments found;
                    warm_first_guesses(S, H, k_all, inv_span, fits, needI, needII, &found, gI, gII);
                    mom = found;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        if (needI) pI[a] = gI[a];
                        if (needII) pII[a] = gII[a];
                    }
                } else {
                    weight_moments(S, H, k_all, inv_span, fits, mom);
                }
            }
            sweep_at(fits, fits);
            const bool redo = fits && ((wmask >> fam) & 1u) && !sums.usable;
            if (__any_sync(kFull, redo)) level_range(S, H, k_all, nz);
            if (kTeam && redo) {   // the same in all lanes of the family's warps
                first_guesses(S, H, k_all, inv_span, nz.ymin, nz.ymax, fits, wantsI, wantsII, mom, pI, pII);
                sweep_at(fits, fits);
                spent = 1;
            } else if (!kTeam && __any_sync(kFull, redo)) {   // rare: kept out of line, with its own copies of what it changes
                double tI[4], tII[4];
#pragma unroll
                for (int a = 0; a < 4; ++a) tI[a] = pI[a], tII[a] = pII[a];
                SweepSums again = sums;
                restart_from_first_guesses(S, fam, H, k_all, inv_span, nz.ymin, nz.ymax, fits, redo, tI, tII, &again);
#pragma unroll
                for (int a = 0; a < 4; ++a) pI[a] = tI[a], pII[a] = tII[a];
                sums = again;
                spent = redo ? 1 : 0;
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) F.p[a] = fam ? pII[a] : pI[a];
        F.ok = fits && sums.usable;
        F.S = sums.S;
        F.lambda = kLambda0;
        F.nu = 2.0;
        F.was_frozen = 0;
        F.sweeps = fits ? 1 + spent : 0;
        F.done = !F.ok;
        F.has_trial = false;
        F.inv_predicted = 0.0;
        park_sums(true);
        SLAQ_PHASE(1);   // first guesses and the sweep at the starting points
        const double tiny_S = 1e-28 * mom.swy2;
        for (int t = 0; t < lm_trials; ++t) {
            if (!__any_sync(kFull, !F.done)) break;
            {
                Sym4 A;
                double gr[4], trial[4] = {0.0, 0.0, 0.0, 0.0};
                normal_equations(S, fam, mom.sw, A, gr);
                prepare_trial<kRows>(F, fam, A, gr, !F.done, tiny_S, span / pitch, trial);
#pragma unroll
                for (int a = 0; a < 4; ++a) {   // each lane of a pair fetches the other family's trial point
                    pI[a] = kTeam ? trial[a] : __shfl_sync(kFull, trial[a], even);
                    pII[a] = kTeam ? trial[a] : a < 3 ? __shfl_sync(kFull, trial[a], oddl) : 0.0;
                }
            }
            const unsigned trying = __ballot_sync(kFull, F.has_trial);
            SLAQ_PHASE(2);   // solver step of a trial
            if (!trying) continue;
            // the lane's own trial point is one of the two it swept: not kept a second time across the sweep
#define SLAQ_OWN_TRIAL {fam ? pII[0] : pI[0], fam ? pII[1] : pI[1], fam ? pII[2] : pI[2], fam ? 0.0 : pI[3]}
            if (kTeam || t + 1 < lm_trials) {
                sweep_at((trying >> even) & 1u, (trying >> oddl) & 1u);
                const double trial[4] = SLAQ_OWN_TRIAL;
                park_sums(finish_trial(F, trial, sums.usable, sums.S));
            } else {   // no step follows: the objective decides, the normal equations are not needed
                bool usable;
                double objective;
                sweep_objective(S, fam, H, k_all, inv_span, pI, pII, usable, objective);
                const double trial[4] = SLAQ_OWN_TRIAL;
                finish_trial(F, trial, usable, objective);
            }
#undef SLAQ_OWN_TRIAL
            SLAQ_PHASE(3);   // sweep at the trial points, reduction, accept or reject
        }
        // both results of the job, in every lane
        double S_I, S_II;
        bool ok_I, ok_II;
        if constexpr (kTeam) {   // through shared memory; the whole block is on this job
            __syncthreads();
            if (lane == 0 && team.part == 0) {
                double* const mine = team.exchange + 16 * fam;
                mine[0] = F.S;
                mine[1] = F.ok ? 1.0 : 0.0;
                mine[2] = (double)F.sweeps;
#pragma unroll
                for (int a = 0; a < 4; ++a) mine[3 + a] = F.p[a];
            }
            __syncthreads();
            const double *const one = team.exchange, *const two = team.exchange + 16;
            S_I = one[0], S_II = two[0];
            ok_I = one[1] > 0.0, ok_II = two[1] > 0.0;
            sweeps_out[0] = (int)one[2], sweeps_out[1] = (int)two[2];
#pragma unroll
            for (int a = 0; a < 4; ++a) pI[a] = one[3 + a], pII[a] = two[3 + a];
        } else {
            S_I = __shfl_sync(kFull, F.S, even), S_II = __shfl_sync(kFull, F.S, oddl);
            ok_I = __shfl_sync(kFull, (int)F.ok, even), ok_II = __shfl_sync(kFull, (int)F.ok, oddl);
            sweeps_out[0] = __shfl_sync(kFull, F.sweeps, even);
            sweeps_out[1] = __shfl_sync(kFull, F.sweeps, oddl);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                pI[a] = __shfl_sync(kFull, F.p[a], even);
                pII[a] = __shfl_sync(kFull, F.p[a], oddl);
            }
        }
        if (kRows) rescale(pI, pII, span / pitch);   // back to the window's coordinates
        if (fits) {
            if (ok_I) S_out[0] = S_I;
            if (ok_II) S_out[1] = S_II;
            const bool okI = ok_I && finite_d(S_I), okII = ok_II && finite_d(S_II);
            ended = (okI ? 1 : 0) | (okII ? 2 : 0);
            // Kept as a flag of its own: a branch on `ended` placed here was compiled as never taken (nvcc 12.9,
            // also with ptxas -O1) although the same value, stored below, is non-zero; a branch on okI || okII is taken.
            any_ended = okI || okII;
#pragma unroll
            for (int a = 0; a < 4; ++a) both_out[a] = pI[a], both_out[4 + a] = pII[a];
            if (okI && (!okII || S_I <= S_II)) {   // a tie goes to family I
                family = 0;
#pragma unroll
                for (int a = 0; a < 4; ++a) p_out[a] = pI[a];
            } else if (okII) {
                family = 1;
#pragma unroll
                for (int a = 0; a < 4; ++a) p_out[a] = pII[a];
            }
        } else {
            sweeps_out[0] = sweeps_out[1] = 0;
        }
    }
    const bool fit_failed = fits && family < 0;
    double rho = nz.rho;
    if (__any_sync(kFull, fit_failed)) {   // rare: the whole warp walks its windows once more
        const double from_levels = mean_change_of_levels(S, H, k_all);
        if (fit_failed) rho = from_levels;
    }
    if (status == SLAQ_JOB_NEW) {
        p_out[0] = 1.0;   // one normalised unit per iteration
        p_out[1] = 1.0;   // at most the whole normalised loss
    } else if (status == SLAQ_JOB_FITTED && family < 0) {
        status = H >= min_fit_points ? SLAQ_JOB_FIT_FAILED : SLAQ_JOB_SHORT;
        const double y_new = S.holds(S.y + lane - S.l) ? S.y[lane - S.l] : 0.0;
        p_out[0] = rho;
        p_out[1] = y_new > 0.0 ? y_new : CUDART_INF;
        p_out[2] = p_out[3] = CUDART_NAN;
    }
    {   // the slot's share of the statistics, one entry per lane
        const bool own = leader && S.l == 0 && H > 0, curve = own && status == SLAQ_JOB_FITTED;
        const unsigned points = __reduce_add_sync(kFull, own ? (unsigned)H : 0u);
        const unsigned swept = __reduce_add_sync(kFull, own ? (unsigned)H * (unsigned)(sweeps_out[0] + sweeps_out[1]) : 0u);
        const unsigned sub = __ballot_sync(kFull, curve && family == 0), expo = __ballot_sync(kFull, curve && family == 1);
        const unsigned other = __ballot_sync(kFull, own && (status == SLAQ_JOB_SHORT || status == SLAQ_JOB_NEW || status == SLAQ_JOB_FIT_FAILED));
        // 1/(a x^2 + b x + c) is convex for all x >= 0 exactly when b^2 >= a c
        const unsigned bent = __ballot_sync(kFull, curve && family == 0 && p_out[1] * p_out[1] < p_out[0] * p_out[2]);
        if (leader && lane < 6)
            tally[lane] += lane == 0 ? points : lane == 1 ? swept : __popc(lane == 2 ? sub : lane == 3 ? expo : lane == 4 ? other : bent);
    }
    if (leader && S.l == 0 && H > 0) {
        fit.status[j] = status;
        fit.mask[j] = (uint8_t)ended;
        if (any_ended) {   // what the next epoch may start from
            fit.k_fit[j] = job.k_last[j];
#pragma unroll
            for (int a = 0; a < 8; ++a) fit.both[8 * (size_t)j + a] = both_out[a];
        }
        fit.family[j] = (int8_t)family;
#pragma unroll
        for (int a = 0; a < 4; ++a) fit.params[4 * (size_t)j + a] = p_out[a];
        fit.residual[2 * (size_t)j] = S_out[0];
        fit.residual[2 * (size_t)j + 1] = S_out[1];
        fit.sweeps[2 * (size_t)j] = sweeps_out[0];
        fit.sweeps[2 * (size_t)j + 1] = sweeps_out[1];
        fit.largest[j] = nz.M;
        fit.span[j] = span;
    }
    __syncwarp();
    SLAQ_PHASE(4);   // winner, fallback, the job's record
}

// kL: lanes per job if the launch has one length class - every cluster with windows of up to about 80 points, or with
// few jobs; 0 where several classes share the launch, each then runs its own instance of fit_slot.
// kRows: false for warm starts (see rescale), and where one warp takes the place of a team of one and has to add as it does.
template <bool kWarm, int kL, int kWarps, bool kRows = !kWarm>
__global__ void __launch_bounds__(kWarps * 32, 1)
fit_kernel(JobArrays job, FitArrays fit, const double* __restrict__ g_wtab, const int32_t* __restrict__ order,
           const int32_t* __restrict__ start, FitClasses cls, int lm_trials, int min_fit_points,
           unsigned int* queue, long long* counters, long long* stamp, int32_t* err_word) {
    extern __shared__ double smem[];
    __shared__ int slot_base[kMaxFitClasses + 1], dealt;
    __shared__ unsigned long long tally[kWarps][6];   // statistics of a warp's jobs, out of its registers
    double* wtab = smem;                                   // [h_max]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* const slice = smem + cls.h_max + (size_t)warp * cls.slice;   // this warp's: parked sums, then the window rows
    for (int i = threadIdx.x; i < cls.h_max; i += blockDim.x) wtab[i] = g_wtab[i];
    if (lane < 6) tally[warp][lane] = 0;
    after_previous();
    note_time(stamp);
    if (threadIdx.x == 0) {   // queue slots of each class: one slot = one warp's worth of jobs
        dealt = 0;
        int run = 0;
        for (int c = 0; c < cls.n; ++c) {
            slot_base[c] = run;
            const int jobs = order ? start[cls.h_lo[c]] - start[cls.h_hi[c]] : job.max_jobs, per_slot = 32 / cls.L[c];
            run += (jobs + per_slot - 1) / per_slot;
        }
        for (int c = cls.n; c <= kMaxFitClasses; ++c) slot_base[c] = run;
    }
    __syncthreads();
    Phases phases = {};
    SLAQ_PHASES_START(phases);
    // The first slots are dealt out to the SMs in turn: slots are sorted by length, and the warps of a block, which draw
    // together, would get neighbours - the longest windows all on one SM (4,000 windows of up to 200 at 16 lanes: 133 us
    // drawn, 113 dealt).  The rest are drawn.
    for (;;) {
        int slot = 0;
        if (lane == 0) {
            const int i = atomicAdd(&dealt, 1), warps = blockDim.x >> 5;
            slot = i < warps ? i * (int)gridDim.x + (int)blockIdx.x : warps * (int)gridDim.x + (int)atomicAdd(queue, 1u);
        }
        slot = __shfl_sync(kFull, slot, 0);
        SLAQ_PHASE(5);   // between jobs: statistics, record tail, queue
        if (slot >= slot_base[cls.n]) break;
        int c = 0;
        while (slot >= slot_base[c + 1]) ++c;
        const int place = slot - slot_base[c];
        switch (kL ? kL : cls.L[c]) {
#define SLAQ_SLOT(n)                                                                                                              \
    case n:                                                                                                                       \
        if constexpr (kL == 0 || kL == n)                                                                                         \
            fit_slot<kWarm, n, kRows, kWarps == 8 ? 2 : 1>(job, fit, order, start, cls, c, place, lm_trials, min_fit_points, wtab, g_wtab + cls.h_max, slice, \
                               tally[warp], lane, phases, err_word);                                                              \
        break;
            SLAQ_SLOT(2) SLAQ_SLOT(4) SLAQ_SLOT(8) SLAQ_SLOT(16) SLAQ_SLOT(32)
#undef SLAQ_SLOT
        }
    }
    // counters 0, 1: points, points swept; 2: fitted jobs; 3, 4: of family I, II; 5: jobs without a curve; 14: not convex ahead
    if (lane < 6) {
        const unsigned long long v = tally[warp][lane];
        if (v) {
            atomicAdd((unsigned long long*)&counters[lane < 2 ? lane : lane == 5 ? 14 : lane + 1], v);
            if (lane == 2 || lane == 3) atomicAdd((unsigned long long*)&counters[2], v);
        }
    }
#ifdef SLAQ_PHASE_CLOCKS
    if (lane == 0)
        for (int i = 0; i < 6; ++i) atomicAdd((unsigned long long*)&counters[8 + i], (unsigned long long)phases.sum[i]);
#endif
}

// A block per job, for clusters with fewer jobs than the GPU has sub-partitions for: each family has warps of its own
// (see Team).  The chain of a trial is shorter than in one warp that does both (fit of 8 windows of 20: 34 -> 28 us, of 160
// of 40: 38 -> 32, of 8 of 1,000 with four warps per family: 82 -> 56).  kListed: the blocks take the jobs of the work list, for
// handles with many more ids (40 windows of up to 900 among 4,000 ids: 83 -> 61 with the sort).
template <bool kWarm, bool kListed>
__global__ void __launch_bounds__(kTeamWarps * 32)
fit_team_kernel(JobArrays job, FitArrays fit, const double* __restrict__ g_wtab, const int32_t* __restrict__ order,
                const int32_t* __restrict__ start, FitClasses cls, int parts, int lm_trials, int min_fit_points,
                long long* counters, long long* stamp, int32_t* err_word) {
    extern __shared__ double smem[];
    __shared__ double exchange[2 * 2 * 4 * 16];
    __shared__ unsigned long long tally[6];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int i = threadIdx.x; i < cls.h_max; i += blockDim.x) smem[i] = g_wtab[i];
    if (threadIdx.x < 6) tally[threadIdx.x] = 0;
    after_previous();
    note_time(stamp);
    __syncthreads();
    Team team;
    team.parts = parts;
    team.shift = 5 + (parts >> 1);   // 1, 2, 4 parts: 32, 64, 128 lanes
    team.fam = warp & 1;
    team.part = warp >> 1;
    const int index = team_index(lane & 15);
    team.index = lane < 16 && index < kParked ? index : -1;
    team.turn = 0;
    team.exchange = exchange;
    Phases phases = {};
    SLAQ_PHASES_START(phases);
    double* const slice = smem + cls.h_max + (size_t)warp * cls.slice;
    if constexpr (kListed) {
        const int jobs = start[0];   // the active ones, at the front of the list
        for (int place = blockIdx.x; place < jobs; place += gridDim.x) {
            fit_slot<kWarm, 32, false, 1, true>(job, fit, order, start, cls, 0, place, lm_trials, min_fit_points, smem, g_wtab + cls.h_max, slice,
                                      tally, lane, phases, err_word, team);
            __syncthreads();   // the exchanged results are read before the next job's are written
        }
    } else {
        fit_slot<kWarm, 32, false, 1, true>(job, fit, nullptr, nullptr, cls, 0, blockIdx.x, lm_trials, min_fit_points, smem, g_wtab + cls.h_max, slice,
                                  tally, lane, phases, err_word, team);
    }
    if (warp == 0 && lane < 6 && tally[lane]) {
        atomicAdd((unsigned long long*)&counters[lane < 2 ? lane : lane == 5 ? 14 : lane + 1], tally[lane]);
        if (lane == 2 || lane == 3) atomicAdd((unsigned long long*)&counters[2], tally[lane]);
    }
#ifdef SLAQ_PHASE_CLOCKS
    if (lane == 0)
        for (int i = 0; i < 6; ++i) atomicAdd((unsigned long long*)&counters[8 + i], (unsigned long long)phases.sum[i]);
#endif
}

// Normalisation only, written out for inspection: same staging and scaling code as the fit,
// one warp per listed job.
__global__ void __launch_bounds__(kMaxWarpsPerBlock * 32)
normalise_export_kernel(JobArrays job, const int32_t* __restrict__ ids, const int64_t* __restrict__ offsets, int n,
                        const double* __restrict__ g_wtab, int max_hist, double* changes, double* levels,
                        double* largest, int32_t* err_word) {
    extern __shared__ double smem[];
    double* wtab = smem;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k_cap = (max_hist + 31) / 32;
    LanesOf<32> S;
    S.y = smem + max_hist + (size_t)warp * (k_cap + 1) * 32;
    S.slice = S.y;
    S.slice_len = (k_cap + 1) * 32;
    S.wtab_len = max_hist;
    S.err_word = err_word;
    S.park = nullptr;
    S.wtab = wtab;
    S.lane = lane;
    S.any_L = 32;
    S.l = lane;
    for (int i = threadIdx.x; i < max_hist; i += blockDim.x) wtab[i] = g_wtab[i];
    __syncthreads();
    const int slot = blockIdx.x * (blockDim.x >> 5) + warp;
    if (slot >= n) return;
    int j = ids[slot];
    if (!index_ok(j, job.max_jobs, kErrJob, err_word)) j = -1;
    const int H = stage_window(job, j, max_hist, S, err_word);
    __syncwarp();
    if (H <= 0) {
        if (lane == 0 && largest) largest[slot] = CUDART_NAN;
        return;
    }
    const int64_t base = offsets[slot];
    const int k_all = (H + 31) / 32;
    const Normalised nz = normalise_window<false>(S, H, k_all, job.m_seen[j], 0, changes ? changes + base : nullptr);
    if (lane == 0 && largest) largest[slot] = nz.M;
    for (int k = 0; k < k_all; ++k) {
        const int m = lane + 32 * k;
        if (m < H) {
            if (nz.status != SLAQ_JOB_FITTED) {   // nothing was scaled: report NaN levels and changes
                if (levels) levels[base + H - 1 - m] = CUDART_NAN;
                if (changes) changes[base + H - 1 - m] = CUDART_NAN;
            } else if (levels) {
                levels[base + H - 1 - m] = S.level(k);
            }
        }
    }
}

// ---- work list: job ids sorted by window length, longest first (counting sort) ----

// Jobs per window length.  Many jobs share a length (a full ring), so lengths are first counted
// in shared memory, lanes with equal lengths adding once, and each block then adds its non-zero
// bins to the global table.
constexpr int kSortThreads = 256;
constexpr int kSortJobsPerBlock = 2048;

__device__ __forceinline__ int clamped_length(const int32_t* __restrict__ count, int j, int max_hist) {
    const int H = count[j];
    return H < 0 ? 0 : (H > max_hist ? max_hist : H);
}

__global__ void __launch_bounds__(kSortThreads)
length_count_kernel(const int32_t* __restrict__ count, int max_jobs, int max_hist, int32_t* bucket, long long* stamp) {
    extern __shared__ int sh_count[];   // [max_hist + 1]
    after_previous();
    note_time(stamp);
    for (int i = threadIdx.x; i <= max_hist; i += blockDim.x) sh_count[i] = 0;
    __syncthreads();
    const int lo = blockIdx.x * kSortJobsPerBlock, hi = min(lo + kSortJobsPerBlock, max_jobs);
    for (int base = lo; base < hi; base += blockDim.x) {
        const int j = base + threadIdx.x;
        const bool in = j < hi;
        const int H = in ? clamped_length(count, j, max_hist) : 0;
        const unsigned live = __ballot_sync(kFull, in);
        if (in) {
            const unsigned peers = __match_any_sync(live, H);
            if ((int)(__ffs(peers) - 1) == (int)(threadIdx.x & 31)) atomicAdd(&sh_count[H], __popc(peers));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= max_hist; i += blockDim.x) {
        const int v = sh_count[i];
        if (v) atomicAdd(&bucket[i], v);
    }
}

// start[h] = number of jobs with a window longer than h (h = 0..max_hist); cursor = copy for the scatter.
__global__ void __launch_bounds__(1024) length_scan_kernel(const int32_t* __restrict__ bucket, int max_hist,
                                                           int32_t* start, int32_t* cursor) {
    __shared__ int sh[1024];
    after_previous();
    const int t = threadIdx.x, n = max_hist + 1;
    const int per = (n + 1023) / 1024;
    // thread t owns lengths h = max_hist - (t * per + i): it walks from the longest down
    int sum = 0;
    for (int i = 0; i < per; ++i) {
        const int h = max_hist - (t * per + i);
        if (h >= 0) sum += bucket[h];
    }
    sh[t] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int v = t >= o ? sh[t - o] : 0;
        __syncthreads();
        sh[t] += v;
        __syncthreads();
    }
    int run = sh[t] - sum;   // jobs longer than this thread's first length
    for (int i = 0; i < per; ++i) {
        const int h = max_hist - (t * per + i);
        if (h < 0) break;
        start[h] = run;
        cursor[h] = run;
        run += bucket[h];
    }
}

// Scatter: a block counts its jobs per length again, reserves one contiguous range per non-zero
// length with a single global atomic, and places its jobs inside those ranges.
__global__ void __launch_bounds__(kSortThreads)
length_scatter_kernel(const int32_t* __restrict__ count, int max_jobs, int max_hist, int32_t* cursor,
                      int32_t* order, int32_t* err_word) {
    extern __shared__ int sh_sort[];    // [max_hist + 1] counts, then [max_hist + 1] next free position
    int* sh_count = sh_sort;
    int* sh_next = sh_sort + (max_hist + 1);
    after_previous();
    for (int i = threadIdx.x; i <= max_hist; i += blockDim.x) sh_count[i] = 0;
    __syncthreads();
    const int lo = blockIdx.x * kSortJobsPerBlock, hi = min(lo + kSortJobsPerBlock, max_jobs);
    const int lane = threadIdx.x & 31;
    for (int base = lo; base < hi; base += blockDim.x) {
        const int j = base + threadIdx.x;
        const bool in = j < hi;
        const int H = in ? clamped_length(count, j, max_hist) : 0;
        const unsigned live = __ballot_sync(kFull, in);
        if (in) {
            const unsigned peers = __match_any_sync(live, H);
            if ((int)(__ffs(peers) - 1) == lane) atomicAdd(&sh_count[H], __popc(peers));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i <= max_hist; i += blockDim.x) {
        const int v = sh_count[i];
        sh_next[i] = v ? atomicAdd(&cursor[i], v) : 0;
    }
    __syncthreads();
    for (int base = lo; base < hi; base += blockDim.x) {
        const int j = base + threadIdx.x;
        const bool in = j < hi;
        const int H = in ? clamped_length(count, j, max_hist) : 0;
        const unsigned live = __ballot_sync(kFull, in);
        if (in) {
            const unsigned peers = __match_any_sync(live, H);
            const int leader = __ffs(peers) - 1;
            int first = 0;
            if (lane == leader) first = atomicAdd(&sh_next[H], __popc(peers));
            first = __shfl_sync(peers, first, leader);
            const int at = first + __popc(peers & ((1u << lane) - 1u));
            if (index_ok(at, max_jobs, kErrJob, err_word)) order[at] = j;
        }
    }
}

// The same in one block for few jobs: count, scan and scatter in shared memory.
constexpr int kOneBlockSort = 16384;

__global__ void __launch_bounds__(1024) length_sort_kernel(const int32_t* __restrict__ count, int max_jobs, int max_hist,
                                                           int32_t* start, int32_t* order, long long* stamp, int32_t* err_word) {
    extern __shared__ int sh_one[];     // [max_hist + 1] jobs per length, then [max_hist + 1] next free position
    __shared__ int warp_sum[32];
    int* const bins = sh_one;
    int* const next = sh_one + (max_hist + 1);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31, n = max_hist + 1;
    for (int i = t; i < n; i += 1024) bins[i] = 0;
    __syncthreads();
    after_previous();
    note_time(stamp);
    int H[kOneBlockSort / 1024];
#pragma unroll
    for (int k = 0; k < kOneBlockSort / 1024; ++k) {
        const int j = k * 1024 + t;
        H[k] = j < max_jobs ? clamped_length(count, j, max_hist) : -1;
    }
#pragma unroll
    for (int k = 0; k < kOneBlockSort / 1024; ++k) {
        if (k * 1024 >= max_jobs) break;
        const unsigned peers = __match_any_sync(kFull, H[k]);
        if (H[k] >= 0 && __ffs(peers) - 1 == lane) atomicAdd(&bins[H[k]], __popc(peers));
    }
    __syncthreads();
    // thread t owns lengths max_hist - (t * per + i): from the longest down, the jobs before its first length
    const int per = (n + 1023) / 1024;
    int sum = 0;
    for (int i = 0; i < per; ++i) {
        const int h = max_hist - (t * per + i);
        if (h >= 0) sum += bins[h];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += up;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int run = incl - sum;
    for (int i = 0; i < warp; ++i) run += warp_sum[i];
    for (int i = 0; i < per; ++i) {
        const int h = max_hist - (t * per + i);
        if (h < 0) break;
        start[h] = run;
        next[h] = run;
        run += bins[h];
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kOneBlockSort / 1024; ++k) {
        if (k * 1024 >= max_jobs) break;
        const unsigned peers = __match_any_sync(kFull, H[k]);
        const int leader = __ffs(peers) - 1;
        int first = 0;
        if (H[k] >= 0 && lane == leader) first = atomicAdd(&next[H[k]], __popc(peers));
        first = __shfl_sync(kFull, first, leader);
        const int at = first + __popc(peers & ((1u << lane) - 1u));
        if (H[k] >= 0 && index_ok(at, max_jobs, kErrJob, err_word)) order[at] = k * 1024 + t;
    }
}

size_t fit_smem_bytes(const FitClasses& c, int warps) {
    return sizeof(double) * ((size_t)c.h_max + (size_t)warps * (size_t)c.slice);
}

}  // namespace

using FitKernel = decltype(&fit_kernel<false, 0, 12>);
using FitTeamKernel = decltype(&fit_team_kernel<false, false>);
// [warps][warm start][lanes: 0 for several, 2, 4, .. 32]; null: never chosen
#define SLAQ_SOME(warm, w) fit_kernel<warm, 2, w>, fit_kernel<warm, 4, w>, fit_kernel<warm, 8, w>, fit_kernel<warm, 16, w>, fit_kernel<warm, 32, w>
static FitKernel const kFitKernels[3][2][6] = {
    {{nullptr, fit_kernel<false, 2, 16>}, {nullptr, fit_kernel<true, 2, 16>}},
    {{fit_kernel<false, 0, 12>, SLAQ_SOME(false, 12)}, {fit_kernel<true, 0, 12>, SLAQ_SOME(true, 12)}},
    {{nullptr, SLAQ_SOME(false, 8)}, {nullptr, SLAQ_SOME(true, 8)}}};
#undef SLAQ_SOME
static FitKernel const kFitAsTeam[2] = {fit_kernel<false, 32, 8, false>, fit_kernel<true, 32, 8, false>};   // see fit_kernel

static FitTeamKernel const kFitTeamKernels[2][2] = {{fit_team_kernel<false, false>, fit_team_kernel<false, true>},
                                                    {fit_team_kernel<true, false>, fit_team_kernel<true, true>}};

// Shared memory beyond the default is allowed to a kernel when a handle is about to use it, which also loads the kernel.  Doing all 26
// in every new handle cost the first one of a process 3 ms more and the later ones 5 us.  The handle remembers the last one: a context
// that is gone takes its handles along.
static cudaError_t allow_shared(slaq_handle* h, const void* kernel, size_t bytes) {
    if (h->fit_ready == kernel) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) h->fit_ready = kernel;
    return e;
}

// active: the handle's active jobs, or as many as it may come to have
static long long jobs_for_lanes(const slaq_handle* h, long long active) {
    return h->fit_cluster_jobs > 0 ? (long long)h->fit_cluster_jobs : active;
}

static int team_slice(const slaq_handle* h) { return kParked * 2 + ((h->max_hist + 31) / 32 + 1) * 32; }
static size_t team_smem(const slaq_handle* h, int parts) {
    return sizeof(double) * ((size_t)h->max_hist + 2 * (size_t)parts * team_slice(h));
}

static FitPlan plan_of(const slaq_handle* h, long long active) {
    return fit_plan(h->max_hist, jobs_for_lanes(h, active), h->sm_count, h->fit_slice_bytes);
}
int fit_least_lanes(const slaq_handle* h) { return plan_of(h, h->n_active).lanes; }

// Warps per family of a job's team; 0: no teams.  A question of the cluster's active jobs and the windows alone, which every shard
// answers alike, whatever its capacity: several warps add in another order than one, and one in another than a part of one.  With a warp per sub-partition at most, a lane is left four rows of the longest
// window; two warps share a sub-partition without loss where a lane would have twelve rows or more (140 windows of up to
// 1,000: 61 -> 58 us, but 200 of up to 300: 44 -> 45), and teams of one warp per family up to sixteen rows (580 windows of 20: 38 ->
// 35 us, but 300 of 1,000: 84 -> 87).
static int fit_team_parts(const slaq_handle* h, long long active) {
    const long long warps = 4LL * h->sm_count, jobs = std::max({1LL, jobs_for_lanes(h, active), active});
    if (2 * jobs > (h->max_hist > 512 ? warps : 2 * warps)) return 0;
    int parts = 1;
    while (parts < kTeamWarps / 2 && ((4 * parts * jobs <= warps && h->max_hist > 128 * parts) ||
                                      (4 * parts * jobs <= 2 * warps && h->max_hist > 384 * parts)))
        parts *= 2;
    while (parts > 0 && team_smem(h, parts) > kTeamSmem) parts >>= 1;
    return parts;
}

// The work list: job ids, longest window first.  Up to kOneBlockSort jobs one block sorts (one launch of about 5 us
// instead of three of 3 to 4 us each), beyond that a block per 2048 jobs.
static cudaError_t launch_sort(slaq_handle* h, cudaStream_t st, int* launches) {
    const int J = h->max_jobs, Hmax = h->max_hist;
    const size_t bins = sizeof(int) * ((size_t)Hmax + 1);
    long long* const stamp = h->scratch.stamps;
    static_assert(2 * sizeof(int) * (kMaxHistLimit + 1) + 32 * sizeof(int) <= 48 * 1024, "both sorts take what a block may use without asking");
    if (J <= kOneBlockSort) {
        *launches += 1;
        return launch_behind(length_sort_kernel, 1, 1024, 2 * bins, st, h->job.count, J, Hmax, h->scratch.start, h->scratch.order, stamp,
                             h->err_word);
    }
    const int sort_blocks = (J + kSortJobsPerBlock - 1) / kSortJobsPerBlock;
    *launches += 3;
    cudaError_t e = launch_behind(length_count_kernel, sort_blocks, kSortThreads, bins, st, h->job.count, J, Hmax, h->scratch.bucket, stamp);
    if (e == cudaSuccess) e = launch_behind(length_scan_kernel, 1, 1024, 0, st, h->scratch.bucket, Hmax, h->scratch.start, h->scratch.cursor);
    if (e == cudaSuccess)
        e = launch_behind(length_scatter_kernel, sort_blocks, kSortThreads, 2 * bins, st, h->job.count, J, Hmax, h->scratch.cursor,
                          h->scratch.order, h->err_word);
    return e;
}

// What a launch of so many active jobs is made of.
struct FitChoice {
    FitClasses cls;
    int parts;      // warps per family of a job's team; 0: fit_kernel
    bool listed;    // the teams take their jobs from the work list
    int warps;      // of a block, at most
    const void* kernel;
    FitKernel fit;
    FitTeamKernel team;
};
static FitChoice fit_choice(const slaq_handle* h, long long active) {
    const int J = h->max_jobs, Hmax = h->max_hist, warm = h->warm_start ? 1 : 0;
    FitChoice c = {};
    c.cls.h_max = Hmax;
    const int parts = fit_team_parts(h, active);
    // A block for each id is for handles with few of them: the empty ones cost 8 jobs among 592 ids 10 us.  A family with one
    // warp adds its sums in the order in which one warp does both, so that teams of one are left to the other kernel there.
    c.listed = J > 4 * h->sm_count;
    if (parts > 1 || (parts == 1 && !c.listed)) {
        c.parts = parts;
        c.cls.n = 1;
        c.cls.h_hi[0] = Hmax;
        c.cls.L[0] = 32;
        c.cls.slice = team_slice(h);
        c.team = kFitTeamKernels[warm][c.listed ? 1 : 0];
        c.kernel = (const void*)c.team;
        return c;
    }
    const FitPlan plan = parts == 1 ? FitPlan{kEight, 32, kFitSlices[kEight]} : plan_of(h, active);
    c.warps = kFitWarps[plan.kind];
    c.cls = fit_classes(Hmax, plan);
    c.fit = parts == 1 ? kFitAsTeam[warm] : kFitKernels[plan.kind][warm][c.cls.n == 1 ? __builtin_ctz((unsigned)c.cls.L[0]) : 0];
    c.kernel = (const void*)c.fit;
    return c;
}

int fit_prepare(slaq_handle* h) {
    const FitChoice c = fit_choice(h, h->max_jobs);
    return allow_shared(h, c.kernel, c.parts ? kTeamSmem : kSmemLimit) == cudaSuccess ? 0 : -1;
}

int launch_fit(slaq_handle* h, cudaStream_t st, int max_blocks) {
    const int J = h->max_jobs;
    int launches = 0;
    const FitChoice c = fit_choice(h, h->n_active);
    const FitClasses& cls = c.cls;
    cudaError_t e = allow_shared(h, c.kernel, c.parts ? kTeamSmem : kSmemLimit);
    if (c.parts) {
        // the list's blocks: one per job that is active now (a graph of the caller's may meet more later)
        const int blocks = c.listed ? std::max(1, h->n_active) : J;
        if (e == cudaSuccess && c.listed) e = launch_sort(h, st, &launches);
        if (e == cudaSuccess)
            e = launch_behind(c.team, blocks, 64 * c.parts, team_smem(h, c.parts), st, h->job, h->fit, h->wtab, h->scratch.order,
                              h->scratch.start, cls, c.parts, h->lm_trials, h->min_fit_points, h->scratch.counters,
                              c.listed ? nullptr : h->scratch.stamps, h->err_word);
        if (e == cudaSuccess) return launches + 1;
        h->err = std::string("fit kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    // A job per warp of the GPU and no more: every job starts at once, so their order means nothing and none is made.
    const bool in_order = cls.n == 1 && cls.L[0] == 32 && J <= max_blocks * c.warps;
    if (e == cudaSuccess && !in_order) e = launch_sort(h, st, &launches);
    // One block per SM: its registers and shared memory fill one.  Where there are fewer slots than warps every SM gets
    // its share of them.
    const long long slots = ((long long)J * cls.L[0] + 31) / 32;   // at most
    const int blocks = (int)std::max(1LL, std::min((long long)max_blocks, slots));
    int warps = c.warps;
    while (warps > 1 && fit_smem_bytes(cls, warps) > kSmemLimit) --warps;
    warps = (int)std::min((long long)warps, (slots + blocks - 1) / blocks);
    // more than half of an SM's shared memory: no SM gets two blocks while another one still holds the kernel before
    const size_t smem = std::max(fit_smem_bytes(cls, warps), kSmemLimit / 2 + 4096);
    if (smem > kSmemLimit) {
        h->err = "fit kernel: a window does not fit in shared memory";
        return -1;
    }
    if (e == cudaSuccess)
        e = launch_behind(c.fit, blocks, warps * 32, smem, st, h->job, h->fit, h->wtab, in_order ? nullptr : h->scratch.order,
                          h->scratch.start, cls, h->lm_trials, h->min_fit_points, h->scratch.ticket + kFitQueueBase, h->scratch.counters,
                          in_order ? h->scratch.stamps : nullptr, h->err_word);
    ++launches;
    if (e != cudaSuccess) {
        h->err = std::string("fit kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return launches;
}

int launch_normalise_export(slaq_handle* h, int32_t n, const int64_t* d_offsets, double* d_changes,
                            double* d_levels, double* d_largest) {
    if (n <= 0) return 0;
    const int k_cap = (h->max_hist + 31) / 32;
    int warps = kMaxWarpsPerBlock;
    auto bytes = [&](int w) { return sizeof(double) * ((size_t)h->max_hist + (size_t)w * (k_cap + 1) * 32); };
    while (warps > 1 && bytes(warps) > kSmemLimit) --warps;
    const size_t smem = bytes(warps);
    cudaError_t e =
        cudaFuncSetAttribute(normalise_export_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) {
        h->err = std::string("normalise kernel shared memory: ") + cudaGetErrorString(e);
        return -1;
    }
    const int blocks = (n + warps - 1) / warps;
    normalise_export_kernel<<<blocks, warps * 32, smem, h->stream>>>(
        h->job, h->stage.ids, d_offsets, n, h->wtab, h->max_hist, d_changes, d_levels, d_largest, h->err_word);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        h->err = std::string("normalise kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

}  // namespace slaq
