// A job's predicted reduction as a function of its cores, shared by the kernel that writes the gain
// table and by the selection that works without one: the iteration-time law, the fitted curve in the
// form the gain formulas need, and the gain of the n-th core.
#pragma once

#include <math_constants.h>

#include "slaq_internal.cuh"

namespace slaq {

namespace gaincurve {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ bool finite_d(double v) { return fabs(v) <= 1.7976931348623157e308; }

// Iteration-time law of job j: the fixed one if set, else ordinary least squares of the
// sampled seconds on u = 1/cores from the running sums.  s and w are left untouched if the
// job has neither; returns whether the law can be used (s >= 0, w > 0, finite).
// kSums: the sums of the samples are loaded with the rest, 64 bytes per job which only few jobs' callers can spare.
template <bool kSums = false>
__device__ inline bool time_law(const JobArrays& job, int j, int max_jobs, double& s, double& w) {
    const double s_fix = job.s_set[j], w_fix = job.w_set[j];
    double early[8];
    if (kSums) {
#pragma unroll
        for (int k = 0; k < 8; ++k) early[k] = job.tm[k * (size_t)max_jobs + j];
    }
    if (finite_d(s_fix) && finite_d(w_fix)) {
        s = s_fix;
        w = w_fix;
    } else {
        const double* tm = job.tm + j;
        const size_t J = (size_t)max_jobs;
        auto sum = [&](int k) { return kSums ? early[k] : tm[k * J]; };
        const double cnt = sum(0), su = sum(1), suu = sum(2), st = sum(3), sut = sum(4), stn = sum(5);
        const double umin = sum(6), umax = sum(7);
        if (!(cnt > 0.0)) return false;
        bool fitted = false;
        if (umax > umin) {
            const double den = __dsub_rn(__dmul_rn(cnt, suu), __dmul_rn(su, su));
            const double ww = __ddiv_rn(__dsub_rn(__dmul_rn(cnt, sut), __dmul_rn(su, st)), den);
            const double ss = __ddiv_rn(__dsub_rn(st, __dmul_rn(ww, su)), cnt);
            if (den > 0.0 && finite_d(ww) && finite_d(ss) && ss >= 0.0 && ww > 0.0) {
                s = ss;
                w = ww;
                fitted = true;
            }
        }
        if (!fitted) {   // one core count only, or an unphysical fit: all time is parallel work
            s = 0.0;
            w = __ddiv_rn(stn, cnt);
        }
    }
    return finite_d(s) && finite_d(w) && w > 0.0 && s >= 0.0;
}

// Reciprocal to about one ulp: hardware seed and two Newton steps.
__device__ __forceinline__ double fast_rcp(double q) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(q));
    double e = fma(-q, x, 1.0);
    x = fma(x, e, x);
    e = fma(-q, x, 1.0);
    return fma(x, e, x);
}

struct Curve {
    int kind;        // 0 family I, 1 family II, 2 linear extrapolation, 3 no gain
    double p0, p1, p2;
    double inv_span, s, w, T;
    double step_scale;   // T w / span: X_n - X_{n-1} = step_scale / ((s n + w)(s (n-1) + w))
};

// Gain of the n-th core.  After an epoch on n cores the job has run m(n) = T n / (s n + w) iterations,
// X_n = m(n) / span in window coordinates.
__device__ inline double raw_gain(const Curve& c, int n) {
    const double den = fma(c.s, (double)n, c.w), denp = fma(c.s, (double)(n - 1), c.w);
    const double inv_den = fast_rcp(den), inv_denp = fast_rcp(denp);
    const double m = c.T * (double)n * inv_den, mp = c.T * (double)(n - 1) * inv_denp;
    const double X = m * c.inv_span, Xp = mp * c.inv_span;
    double gain;
    if (c.kind == 0) {
        // 1/q(Xp) - 1/q(X) = (q(X) - q(Xp)) / (q(X) q(Xp)), q(X) - q(Xp) = (X - Xp)(a (X + Xp) + b)
        const double dX = c.step_scale * inv_den * inv_denp;
        const double q_now = fma(fma(c.p0, X, c.p1), X, c.p2);
        const double q_prev = fma(fma(c.p0, Xp, c.p1), Xp, c.p2);
        const double dq = dX * fma(c.p0, X + Xp, c.p1);
        gain = dq * fast_rcp(q_now * q_prev);
    } else if (c.kind == 1) {
        // e^(alpha - beta Xp) - e^(alpha - beta X) = e^(alpha - beta Xp) (1 - e^(-beta (X - Xp)))
        const double dX = c.step_scale * inv_den * inv_denp;
        gain = exp(fma(-c.p1, Xp, c.p0)) * (-expm1(-c.p1 * dX));
    } else {
        gain = fmin(c.p0 * m, c.p1) - fmin(c.p0 * mp, c.p1);
    }
    return (finite_d(gain) && gain > 0.0) ? gain : 0.0;
}

// T w / span, in one order of its two products wherever a curve is put together.
__device__ __forceinline__ double step_scale_of(double T, double w, double inv_span) { return T * w * inv_span; }

// A curve as it was when its epoch ran.
__device__ __forceinline__ void keep_curve(const GainBasis& b, int j, int max_jobs, const Curve& c, int kind) {
    double* const v = b.v + j;
    const size_t J = (size_t)max_jobs;
    v[0] = c.p0;
    v[J] = c.p1;
    v[2 * J] = c.p2;
    v[3 * J] = c.inv_span;
    v[4 * J] = c.s;
    v[5 * J] = c.w;
    b.kind[j] = (int8_t)kind;
}
__device__ __forceinline__ Curve kept_curve(const GainBasis& b, int j, int max_jobs, double T) {
    const double* const v = b.v + j;
    const size_t J = (size_t)max_jobs;
    Curve c;
    c.p0 = v[0];
    c.p1 = v[J];
    c.p2 = v[2 * J];
    c.inv_span = v[3 * J];
    c.s = v[4 * J];
    c.w = v[5 * J];
    c.kind = b.kind[j];
    c.T = T;
    c.step_scale = step_scale_of(T, c.w, c.inv_span);
    return c;
}

// The curve of job j for this epoch.  Sets kind 3 (no gain) for jobs that predict nothing; a job
// that could predict but has no usable time law gets status SLAQ_JOB_NO_TIME, which the caller
// records (*no_time).
// kEager: all loads are issued before any is used, for callers that wait for every one of them.
template <bool kEager = false, bool kSums = false>
__device__ inline Curve load_curve(const JobArrays& job, const FitArrays& fit, int j, int max_jobs, double T,
                                   bool* no_time) {
    const int status = fit.status[j];
    const bool active = job.count[j] > 0;
    double p[3];
    int family = 0;
    bool law = false;
    Curve c;
    c.s = c.w = 0.0;
    if (kEager) {
#pragma unroll
        for (int k = 0; k < 3; ++k) p[k] = fit.params[4 * (size_t)j + k];
        family = fit.family[j];
        law = time_law<kSums>(job, j, max_jobs, c.s, c.w);
    }
    c.kind = 3;
    c.T = T;
    c.inv_span = 1.0 / fit.span[j];
    c.p0 = c.p1 = c.p2 = c.step_scale = 0.0;
    *no_time = false;
    const bool predicts = status == SLAQ_JOB_FITTED || status == SLAQ_JOB_SHORT || status == SLAQ_JOB_NEW ||
                          status == SLAQ_JOB_FIT_FAILED;
    if (active && status != SLAQ_JOB_NONFINITE && status != SLAQ_JOB_FLAT) {
        if (!(kEager ? law : time_law(job, j, max_jobs, c.s, c.w))) {
            *no_time = true;
        } else if (predicts) {
            c.p0 = kEager ? p[0] : fit.params[4 * (size_t)j];
            c.p1 = kEager ? p[1] : fit.params[4 * (size_t)j + 1];
            c.p2 = kEager ? p[2] : fit.params[4 * (size_t)j + 2];
            c.kind = status == SLAQ_JOB_FITTED ? (kEager ? family : (int)fit.family[j]) : 2;
            c.step_scale = step_scale_of(T, c.w, c.inv_span);
        }
    }
    return c;
}

}  // namespace gaincurve

}  // namespace slaq
