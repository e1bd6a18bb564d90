// The inner loop of the curve fit: one sweep over a job's window that evaluates both
// convergence families of "Predicting Quality Improvement" at their current points and
// accumulates the sums of their normal equations.  Kept in a header of its own so that the
// stand-alone timing program (bench_probes/fit_sweep_probe.cu) runs exactly this code.
#pragma once

#include <math_constants.h>

#include "slaq_bounds.cuh"

namespace slaq {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ bool finite_d(double v) { return fabs(v) <= 1.7976931348623157e308; }

// Reciprocal to about one ulp: hardware seed (2^-20 or better) and one step of third order, x (1 + e + e^2) with
// e = 1 - q x, which takes one instruction fewer than two Newton steps (no special-case paths;
// a zero, subnormal or non-finite argument gives a non-finite or zero result, which the
// callers treat as "not usable").
__device__ __forceinline__ double fast_rcp(double q) {
    double x;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(q));
    const double e = fma(-q, x, 1.0);
    return fma(x, fma(e, e, e), x);
}

// Shared-memory view of one warp.  Point m of a lane's job (m = distance from the newest
// point, m = l + L k for the lane with index l in its group) sits at y[k * 32 + lane]:
// every access of the sweeps is lane-private and free of bank conflicts.
// kL: the lanes per job where all jobs of a launch have the same (a constant for the compiler), else 0.
// kRows: x counts rows of a lane's points (x = -m / L; see rescale), else windows (x = -m / (H - 1)).
// kStep: rows a sweep's walk takes at once, where registers are there for two.
template <int kL, bool kRows = true, int kStep = 1>
struct LanesOf {
    static constexpr int kRowsAtOnce = kStep;
    static constexpr bool kRowUnit = kRows;
    double* y;         // [k_cap + 1][32]
    double* park;      // this lane's family of its job in [kParked][2 * jobs per warp] (one column per job and family)
    const double* wtab;
    const double* wsum;   // in global memory: [5][wtab_len + 1] sums over m < H of gamma^m m^p (first guesses only)
    int lane, l;
    int any_L;         // lanes per job (kL == 0)
    __device__ __forceinline__ int L() const { return kL ? kL : any_L; }
    __device__ __forceinline__ const double* log_table() const { return wsum + 5 * (wtab_len + 1) + 1; }   // see log_of_normal
    __device__ __forceinline__ int park_stride() const { return 64 >> (__ffs(L()) - 1); }   // 2 * (32 / L), L() a power of two
    // Which of its family's 13 sums the lane holds after a sweep's reduction (see halve): `n` of them from the `from`-th on.
    __device__ __forceinline__ void held(int& from, int& n) const {
        from = 0, n = 13;
        if (L() >= 4) { const int b = (lane >> 1) & 1; from = 7 * b; n = 7 - b; }
        if (L() >= 8) { const int b = (lane >> 2) & 1; from += 4 * b; n = b ? n - 4 : 4; }
        if (L() >= 16) { const int b = (lane >> 3) & 1; from += 2 * b; n = b ? max(n - 2, 0) : min(n, 2); }
        if (L() >= 32) { const int b = (lane >> 4) & 1; from += b; n = b ? max(n - 1, 0) : min(n, 1); }
    }
    // Where the steps of the reduction leave the objective, sum 12 of either family.
    __device__ __forceinline__ int objective_lane() const {
        return (lane & -L()) + (lane & 1) + 2 + (L() >= 8 ? 4 : 0) + (L() >= 32 ? 16 : 0);
    }
    __device__ __forceinline__ unsigned group() const {   // the lanes of this lane's job
        return (0xffffffffu >> (32 - L())) << (lane & -L());
    }
    // extents, read by the bounds build only: the warp's slice [slice, slice + slice_len) and the weight table
    const double* slice;
    int slice_len, wtab_len;
    int32_t* err_word;
    __device__ __forceinline__ bool holds(const double* p) const {
        return index_ok(p - slice, slice_len, kErrShared, err_word);
    }
    __device__ __forceinline__ double weight(int m) const {
        return index_ok(m, wtab_len, kErrShared, err_word) ? wtab[m] : 0.0;
    }
    __device__ __forceinline__ double weight(const double* p) const {   // p = wtab + m
        return index_ok(p - wtab, wtab_len, kErrShared, err_word) ? *p : 0.0;
    }
    __device__ __forceinline__ double level(int k) const {   // the lane's point of row k
        const double* p = y + k * 32 + lane;
        return holds(p) ? *p : 0.0;
    }
};

// The window value at distance m + 1 from the newest point, seen from the lane that owns m.
template <class Lanes>
__device__ __forceinline__ double older_neighbour(const Lanes& S, int k) {
    const double* p = S.l + 1 < S.L() ? S.y + k * 32 + S.lane + 1 : S.y + (k + 1) * 32 + S.lane - (S.L() - 1);
    return S.holds(p) ? *p : 0.0;
}

// What a lane keeps of one sweep: its share of the sums of ITS family over the whole window (see LanesOf::held), and the objective.
// Family I (u = 1/q^2, J = (-u x^2, -u x, -u, 1)): v[0..4] = sum w u^2 x^k, v[5..7] = sum w u x^k,
// v[8..10] = sum w u r x^k, v[11] = sum w r, v[12] = S.
// Family II (J = (e, -x e, 1)) has its entries of the normal equations where family I has the same ones, with the sign
// family I's are read with, so that both solvers read one layout: v[4], -v[3], v[2] = sum w e^2 x^k, v[5], -v[1] = sum w e
// x^k, -v[10], v[9] = sum w e r x^k, v[8] = -sum w r, v[12] = S, the others 0.
struct SweepSums {
    double v[13];
    double S;      // the objective
    bool usable;   // the model was defined at every point and all sums are finite
};

// Running sums to sums of powers of u.  A lane walks its points from the oldest to the newest and keeps, for a
// weighted value a, the chain c0 += a, c1 -= c0, c2 -= c1, ... in which every link takes the value its
// predecessor had one step earlier; after the walk c_p = (-1)^p sum a_k C(k, p), k = the row of the point counted from
// the lane's newest.  Powers of k are fixed combinations with positive coefficients (k^2 = 2 C(k,2) + C(k,1),
// k^3 = 6 C(k,3) + 6 C(k,2) + C(k,1), k^4 = 24 C(k,4) + 36 C(k,3) + 14 C(k,2) + C(k,1)); with u = u_l - k
// (u_l <= 0 the lane's newest point) the powers of u follow from a shift of the origin, all of whose terms have the sign
// of (-1)^p: nothing cancels, the sums are as accurate as if the powers had been multiplied out point by point.
template <int P>
__device__ __forceinline__ void chains_to_powers(double (&c)[P], double u_l) {
    const double c1 = P > 1 ? c[1] : 0.0, c2 = P > 2 ? c[2] : 0.0, c3 = P > 3 ? c[3] : 0.0;
    if (P > 2) c[2] = fma(2.0, c2, -c1);
    if (P > 3) c[3] = fma(6.0, c3, fma(-6.0, c2, c1));
    if (P > 4) c[4] = fma(24.0, c[4], fma(-36.0, c3, fma(14.0, c2, -c1)));
#pragma unroll
    for (int j = 1; j < P; ++j)
#pragma unroll
        for (int p = P - 1; p >= j; --p) c[p] = fma(u_l, c[p - 1], c[p]);
}

// The same in a unit in which a row is g long (g < 0), from chains that add: the powers of k are scaled by g^p first.  For warm starts and the
// teams, whose lanes have a row or two: nothing is gained there by counting in rows.
template <int P>
__device__ __forceinline__ void chains_to_powers(double (&c)[P], double x_l, double g) {
    const double c1 = P > 1 ? c[1] : 0.0, c2 = P > 2 ? c[2] : 0.0, c3 = P > 3 ? c[3] : 0.0;
    if (P > 2) c[2] = fma(2.0, c2, c1);
    if (P > 3) c[3] = fma(6.0, c3, fma(6.0, c2, c1));
    if (P > 4) c[4] = fma(24.0, c[4], fma(36.0, c3, fma(14.0, c2, c1)));
    double gp = g;
#pragma unroll
    for (int i = 1; i < P; ++i, gp *= g) c[i] *= gp;
#pragma unroll
    for (int j = 1; j < P; ++j)
#pragma unroll
        for (int p = P - 1; p >= j; --p) c[p] = fma(x_l, c[p - 1], c[p]);
}

// The running sums of one lane: family I (m: w u^2, n: w u, h: w u r, gd: w r, sI: w r^2 with u = 1/q^2) and
// family II (ee: w e^2, f: w e, kk: w e r, gc: w r, sII: w r^2).
struct LaneSums {
    double m[5], n[3], h[3], gd, sI;
    double ee[3], f[2], kk[2], gc, sII;
    int q_signs;     // OR of the high words of family I's denominators: negative if one of them had its sign bit set
};

template <bool kRows>
__device__ __forceinline__ void link(double& c, double before) {
    if (kRows) c -= before;
    else c += before;
}

// One point of a lane's walk: both families' values at the point and their running sums.  kRows: x counts rows (see chains_to_powers).
template <bool kI, bool kII, bool kRows, class Lanes>
__device__ __forceinline__ void add_point(const Lanes& S, const double* wp, const double* yp, double x,
                                          const double (&pI)[4], const double (&pII)[4], double& e, double ratio,
                                          LaneSums& a) {
    const double w = S.weight(wp);
    const double y = S.holds(yp) ? *yp : 0.0;
    if (kI) {
        const double q = fma(fma(pI[0], x, pI[1]), x, pI[2]);
        a.q_signs |= __double2hiint(q);   // q = 0 or NaN makes the sums non-finite, which the caller sees
        const double inv = fast_rcp(q);
        const double r = y - (inv + pI[3]);
        const double u = inv * inv;
        const double wu = w * u, wuu = wu * u, wur = wu * r, wr = w * r;
        link<kRows>(a.m[4], a.m[3]); link<kRows>(a.m[3], a.m[2]); link<kRows>(a.m[2], a.m[1]); link<kRows>(a.m[1], a.m[0]); a.m[0] += wuu;
        link<kRows>(a.n[2], a.n[1]); link<kRows>(a.n[1], a.n[0]); a.n[0] += wu;
        link<kRows>(a.h[2], a.h[1]); link<kRows>(a.h[1], a.h[0]); a.h[0] += wur;
        a.gd += wr;
        a.sI = fma(wr, r, a.sI);
    }
    if (kII) {
        const double r = y - (e + pII[2]);
        const double we = w * e, wee = we * e, wer = we * r, wr = w * r;
        link<kRows>(a.ee[2], a.ee[1]); link<kRows>(a.ee[1], a.ee[0]); a.ee[0] += wee;
        link<kRows>(a.f[1], a.f[0]); a.f[0] += we;
        link<kRows>(a.kk[1], a.kk[0]); a.kk[0] += wer;
        a.gc += wr;
        a.sII = fma(wr, r, a.sII);
        e *= ratio;
    }
}

// The walk over a lane's rows, oldest first.  kI / kII: whether the family is evaluated at all - the same for
// the whole warp, so that the loop has no branch per family (a lane whose family has no trial computes it at
// parameters nobody uses and its sums are discarded).  Branches inside the loop cost issue slots on every row:
// the rows that every lane of the warp has are walked without a test, only the ragged rest with one.
template <bool kI, bool kII, class Lanes>
__device__ __forceinline__ void walk_rows(const Lanes& S, int k_last, int k_all, double inv_span, const double (&pI)[4],
                                          const double (&pII)[4], LaneSums& a) {
    const int mi = S.l + k_last * S.L();
    // in rows x and its steps are exact
    constexpr bool kRows = Lanes::kRowUnit;
    const double md = (double)mi, hx = kRows ? 1.0 : (double)S.L() * inv_span;
    double x = kRows ? md * (-1.0 / (double)S.L()) : -md * inv_span;
    // e = exp(alpha - beta x) falls geometrically towards the newest point: one
    // exact value at the lane's oldest point, then a constant ratio per step.  (Choosing the start such
    // that the recurrence lands on the exact value at the newest point was measured: the predictions stay
    // as close to the reference's either way, and the extra arithmetic costs 2 % of the kernel.)
    double e = 0.0, ratio = 1.0;
    if (kII) {
        e = exp(fma(-pII[1], x, pII[0]));
        ratio = exp(-pII[1] * hx);
    }
    const double* yp = S.y + S.lane + k_last * 32;
    const double* wp = S.wtab + mi;
    const int k_min = __reduce_min_sync(kFull, k_last);
    int i = 0;
#pragma unroll Lanes::kRowsAtOnce
    for (; i <= k_min; ++i, x += hx, yp -= 32, wp -= S.L()) add_point<kI, kII, kRows>(S, wp, yp, x, pI, pII, e, ratio, a);
#pragma unroll 1
    for (; i < k_all; ++i, x += hx, yp -= 32, wp -= S.L())
        if (i <= k_last) add_point<kI, kII, kRows>(S, wp, yp, x, pI, pII, e, ratio, a);   // row k_last - i >= 0
}

// One step of the reduction over the lanes of a group: of N sums a lane keeps the lower K (bit `o` of its number clear) or
// the upper N - K (set), and adds the partner's.
template <int K, int N>
__device__ __forceinline__ void halve(double (&v)[13], int o, int lane) {
    const bool upper = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double hi = K + k < N ? v[K + k] : 0.0;
        const double give = upper ? v[k] : hi;
        v[k] = (upper ? hi : v[k]) + __shfl_xor_sync(kFull, give, o);
    }
}

// One sweep over the window: both families at once, each at its own point.  A lane adds up
// both families over its points, oldest first, as running sums (see chains_to_powers: in the loop
// every accumulation but the two objectives is an addition of two registers, which the fp64 pipe
// issues in two cycles where a fused multiply-add on three registers takes three); the first
// reduction step hands each lane of a pair the other lane's partial sums of its own family, the
// remaining steps run over lanes of the same parity.  With few rows per lane these steps are most of a sweep: exchanging
// all 13 sums in each took 840 of the 5,300 cycles of a trial at 32 lanes and one row per lane.
template <class Lanes>
__device__ __forceinline__ void sweep(const Lanes& S, int fam, int H, int k_all, double inv_span,
                                      const double (&pI)[4], bool doI, const double (&pII)[4], bool doII,
                                      SweepSums& out) {
    LaneSums a = {};
    const int shift = __ffs(S.L()) - 1;                                      // L is a power of two
    const int k_last = H - 1 - S.l >= 0 ? (H - 1 - S.l) >> shift : -1;     // the row of the lane's oldest point
    const bool anyI = __any_sync(kFull, doI), anyII = __any_sync(kFull, doII);
    if (anyI && anyII) {
        walk_rows<true, true>(S, k_last, k_all, inv_span, pI, pII, a);
    } else {   // one family has no trial left in the whole warp
        if (anyI) walk_rows<true, false>(S, k_last, k_all, inv_span, pI, pII, a);
        if (anyII) walk_rows<false, true>(S, k_last, k_all, inv_span, pI, pII, a);
    }
    double (&m)[5] = a.m, (&n)[3] = a.n, (&h)[3] = a.h, (&ee)[3] = a.ee, (&f)[2] = a.f, (&kk)[2] = a.kk;
    const double gd = a.gd, sI = a.sI, gc = a.gc, sII = a.sII;
    if constexpr (Lanes::kRowUnit) {
        const double x_l = (double)S.l * (-1.0 / (double)S.L());
        chains_to_powers(m, x_l), chains_to_powers(n, x_l), chains_to_powers(h, x_l);
        chains_to_powers(ee, x_l), chains_to_powers(f, x_l), chains_to_powers(kk, x_l);
    } else {
        const double x_l = -(double)S.l * inv_span, g = -((double)S.L() * inv_span);
        chains_to_powers(m, x_l, g), chains_to_powers(n, x_l, g), chains_to_powers(h, x_l, g);
        chains_to_powers(ee, x_l, g), chains_to_powers(f, x_l, g), chains_to_powers(kk, x_l, g);
    }
    // pair step: an even lane hands over its family-II partials and receives family-I ones, an odd lane the reverse
    const bool odd = fam != 0;
    double v[13];
#define SLAQ_PAIR(k, a, b) v[k] = (odd ? (b) : (a)) + __shfl_xor_sync(kFull, odd ? (a) : (b), 1)
    SLAQ_PAIR(1, m[1], -f[1]); SLAQ_PAIR(2, m[2], ee[2]); SLAQ_PAIR(3, m[3], -ee[1]); SLAQ_PAIR(4, m[4], ee[0]);
    SLAQ_PAIR(5, n[0], f[0]); SLAQ_PAIR(8, h[0], -gc); SLAQ_PAIR(9, h[1], kk[1]); SLAQ_PAIR(10, h[2], -kk[0]);
    SLAQ_PAIR(12, sI, sII);
#undef SLAQ_PAIR
    // family I only: an odd lane has no such sums
    v[0] = m[0] + __shfl_xor_sync(kFull, m[0], 1);
    v[6] = n[1] + __shfl_xor_sync(kFull, n[1], 1);
    v[7] = n[2] + __shfl_xor_sync(kFull, n[2], 1);
    v[11] = gd + __shfl_xor_sync(kFull, gd, 1);
    if (odd) v[0] = v[6] = v[7] = v[11] = 0.0;
    // Remaining steps over the lanes of the same parity: in each a lane hands over one half of its sums and keeps the
    // other, 7 + 4 + 2 + 1 exchanges instead of 13 in every step, and every sum ends in one lane.
    double chk, objective;
    if (S.L() == 2) {
        // Family I: sum w u^2 and sum w u^2 x^4 bound what lies between, and sum |w u r x^k| <= sqrt(sum w u^2 x^2k . sum w r^2).  Family II:
        // sum w e^2 bounds its sums without x.  Those with x, which counts rows in cold fits and is counted in rows by the chains always, can be
        // up to the square of a lane's rows (9,025 at eight warps) times as large.  Where they overflow and sum w e^2 does not, within four
        // orders of the end of the range, the point stands, no step is found from it and the fit ends there; more lanes drop it.
        objective = v[12];
        chk = (v[0] + v[4]) + v[12];
    } else {
        halve<7, 13>(v, 2, S.lane);
        if (S.L() == 4) {
            objective = v[5];
            chk = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + v[6]);
        } else {
            halve<4, 7>(v, 4, S.lane);
            if (S.L() == 8) {
                objective = v[1];
                chk = (v[0] + v[1]) + (v[2] + v[3]);
            } else {
                halve<2, 4>(v, 8, S.lane);
                objective = v[1];
                chk = v[0] + v[1];
                if (S.L() == 32) {
                    halve<1, 2>(v, 16, S.lane);
                    objective = chk = v[0];
                }
            }
        }
        objective = __shfl_sync(kFull, objective, S.objective_lane());
    }
#pragma unroll
    for (int k = 0; k < 13; ++k) out.v[k] = v[k];
    out.S = objective;
    const unsigned broken = __ballot_sync(kFull, !finite_d(chk)), negative = __ballot_sync(kFull, a.q_signs < 0);
    const unsigned group = S.group();
    out.usable = !(broken & group & (odd ? 0xaaaaaaaau : 0x55555555u)) && (odd || !(negative & group));
}

// A job's team of warps, where there are more warps than jobs: `parts` warps (1, 2 or 4) for each family, which share
// its rows.  Every warp holds the whole window and runs its family's solver on the same sums, so they all decide alike.
struct Team {
    int fam, part, parts, shift;   // 32 parts = 1 << shift lanes in all
    int index;                     // which sum the lane ends with (-1: none that is parked)
    int turn;
    double* exchange;              // [2][2][4][16] in shared memory
};

// Which of the 13 sums a lane holds after the steps of sweep_team (13: none).
__device__ __forceinline__ int team_index(int lane) {
    const int b0 = lane & 1, b1 = lane >> 1 & 1, b2 = lane >> 2 & 1, b3 = lane >> 3 & 1;
    const int at = 4 * b1 + 2 * b2 + b3;
    return b0 ? min(7 + at, 13) : (at < 7 ? at : 13);
}

// One sweep of one family by its team: half the arithmetic per point, no exchange between families, and a lane has
// as few rows as the team has lanes.
template <int kFam>
__device__ __forceinline__ void sweep_team(const LanesOf<32, false>& S, Team& t, int H, double inv_span, const double (&p)[4], SweepSums& out) {
    LaneSums a = {};
    const int LT = 1 << t.shift, lt = S.lane + 32 * t.part;
    const int k_last = H - 1 - lt >= 0 ? (H - 1 - lt) >> t.shift : -1;
    const int k_all = (H + LT - 1) >> t.shift;
    const int mi = lt + k_last * LT;
    const double md = (double)mi, hx = (double)LT * inv_span;
    double x = -md * inv_span, e = 0.0, ratio = 1.0;
    if (kFam == 1) {
        e = exp(fma(p[1], md * inv_span, p[0]));
        ratio = exp(-p[1] * hx);
    }
    const double* yp = S.y + mi;   // point m lies at y[(m / 32) * 32 + lane], and mi is lane + 32 times something
    const double* wp = S.wtab + mi;
#pragma unroll 1
    for (int i = 0; i < k_all; ++i, x += hx, yp -= LT, wp -= LT)
        if (i <= k_last) add_point<kFam == 0, kFam == 1, false>(S, wp, yp, x, p, p, e, ratio, a);
    const double x_l = -(double)lt * inv_span, g = -hx;
    double v[13];
    if (kFam == 0) {
        chains_to_powers(a.m, x_l, g);
        chains_to_powers(a.n, x_l, g);
        chains_to_powers(a.h, x_l, g);
        v[0] = a.m[0]; v[1] = a.m[1]; v[2] = a.m[2]; v[3] = a.m[3]; v[4] = a.m[4];
        v[5] = a.n[0]; v[6] = a.n[1]; v[7] = a.n[2]; v[8] = a.h[0]; v[9] = a.h[1]; v[10] = a.h[2];
        v[11] = a.gd; v[12] = a.sI;
    } else {
        chains_to_powers(a.ee, x_l, g);
        chains_to_powers(a.f, x_l, g);
        chains_to_powers(a.kk, x_l, g);
        v[0] = 0.0; v[1] = -a.f[1]; v[2] = a.ee[2]; v[3] = -a.ee[1]; v[4] = a.ee[0]; v[5] = a.f[0]; v[6] = v[7] = 0.0;
        v[8] = -a.gc; v[9] = a.kk[1]; v[10] = -a.kk[0]; v[11] = 0.0; v[12] = a.sII;
    }
    halve<7, 13>(v, 1, S.lane);
    halve<4, 7>(v, 2, S.lane);
    halve<2, 4>(v, 4, S.lane);
    halve<1, 2>(v, 8, S.lane);
    double own = v[0] + __shfl_xor_sync(kFull, v[0], 16);
    bool negative = kFam == 0 && __any_sync(kFull, a.q_signs < 0);
    if (t.parts > 1) {   // the parts' sums, in the same order in every warp
        double* const at = t.exchange + ((t.turn * 2 + kFam) * 4) * 16;
        t.turn ^= 1;   // the other half next time: a warp may still be reading this one then
        if (S.lane < 16) at[t.part * 16 + S.lane] = S.lane == 15 ? (negative ? 1.0 : 0.0) : own;
        asm volatile("bar.sync %0, %1;" ::"r"(1 + kFam), "r"(LT) : "memory");
        own = at[S.lane & 15];
        for (int q = 1; q < t.parts; ++q) own += at[q * 16 + (S.lane & 15)];
        negative = kFam == 0 && __shfl_sync(kFull, own, 15) > 0.0;
    }
    out.v[0] = own;
    out.S = __shfl_sync(kFull, own, 11);   // where sum 12 ends
    out.usable = __all_sync(kFull, finite_d(own)) && !negative;
}

// The objectives alone, for a trial after which no further step is taken: a third of the sweep's arithmetic per point, and
// nothing to reduce but the objective.  Added up in the sweep's order, so the same to the bit.  A point at which the model
// is not defined makes its objective non-finite or its denominator negative; the other sums are bounded by the
// objective and the finite denominators.
template <class Lanes>
__device__ __forceinline__ void sweep_objective(const Lanes& S, int fam, int H, int k_all, double inv_span,
                                                const double (&pI)[4], const double (&pII)[4], bool& usable, double& objective) {
    const int shift = __ffs(S.L()) - 1;
    const int k_last = H - 1 - S.l >= 0 ? (H - 1 - S.l) >> shift : -1;
    const int mi = S.l + k_last * S.L();
    const double md = (double)mi, hx = Lanes::kRowUnit ? 1.0 : (double)S.L() * inv_span;
    double x = Lanes::kRowUnit ? md * (-1.0 / (double)S.L()) : -md * inv_span;
    double e = exp(fma(-pII[1], x, pII[0]));
    const double ratio = exp(-pII[1] * hx);
    double sI = 0.0, sII = 0.0;
    int q_signs = 0;
    const double* yp = S.y + S.lane + k_last * 32;
    const double* wp = S.wtab + mi;
#pragma unroll 1
    for (int i = 0; i < k_all; ++i, x += hx, yp -= 32, wp -= S.L()) {
        if (i <= k_last) {
            const double w = S.weight(wp);
            const double y = S.holds(yp) ? *yp : 0.0;
            const double q = fma(fma(pI[0], x, pI[1]), x, pI[2]);
            q_signs |= __double2hiint(q);
            const double rI = y - (fast_rcp(q) + pI[3]), rII = y - (e + pII[2]);
            sI = fma(w * rI, rI, sI);
            sII = fma(w * rII, rII, sII);
            e *= ratio;
        }
    }
    const bool odd = fam != 0;
    double v = (odd ? sII : sI) + __shfl_xor_sync(kFull, odd ? sI : sII, 1);
    for (int o = 2; o < S.L(); o <<= 1) v += __shfl_xor_sync(kFull, v, o);
    objective = v;
    const unsigned negative = __ballot_sync(kFull, q_signs < 0);
    usable = finite_d(v) && (odd || !(negative & S.group()));
}

}  // namespace slaq
