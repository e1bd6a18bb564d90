// The logarithm that the first guesses of cold fits take, and its table.  Compiles for the host as well, where its accuracy is tested.
#pragma once

#include <array>
#include <cmath>
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define SLAQ_BOTH __host__ __device__ __forceinline__
#else
#define SLAQ_BOTH inline
#endif

namespace slaq {

constexpr int kLogBins = 128;                             // the table's bins, where they begin and how wide they are
constexpr int kLogFrom = 0x3fe6b000, kLogBinShift = 13;   // in high words; 1 is the middle of bin 74

SLAQ_BOTH int64_t log_bits(double x) {
#ifdef __CUDA_ARCH__
    return __double_as_longlong(x);
#else
    int64_t b;
    std::memcpy(&b, &x, sizeof b);
    return b;
#endif
}
SLAQ_BOTH double log_value(int64_t b) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double(b);
#else
    double x;
    std::memcpy(&x, &b, sizeof x);
    return x;
#endif
}

// log of a positive normal number, to 0.503 ulp, by table lookup (Tang, "Table-driven implementation of the logarithm function", 1990):
// x = 2^e z with z in about [0.71, 1.42) cut into 128 bins with middles c, log x = e log 2 + log c + log(1 + r) with
// r = z / c - 1, |r| <= 2^-8, by its Taylor series.  log 2 and log c are split so that the leading parts add up exactly; the bin
// around 1 has c = 1.  r is kept with what its rounding left, and the leading parts are added to it exactly: beside 1 the logarithm is as
// small as r, and without that the error is 1.24 ulp.  Over 25 million arguments in each of five ranges the error is 0.503 ulp at most, and
// no larger on average than log()'s (0.553 at most).  tab: 128 pairs of 1 / c and the leading part of log c, then the rests.
// Shorter than log(), whose arguments may be anything (fit of 100,000 windows of up to 1,000: 3,520 -> 3,468 us, of
// 1,000,000 of 64: 3,810 -> 3,802).
SLAQ_BOTH double log_of_normal(double x, const double* __restrict__ tab) {
    const int64_t b = log_bits(x);
    const int t = (int)(b >> 32) - kLogFrom, e = t >> 20, bin = (t >> kLogBinShift) & (kLogBins - 1);
    const double z = log_value(b - ((int64_t)e << 52));
#ifdef __CUDA_ARCH__
    const double2 c = __ldg(reinterpret_cast<const double2*>(tab) + bin);
    const double inv = c.x, log_c = c.y, rest = __ldg(tab + 2 * kLogBins + bin);
#else
    const double inv = tab[2 * bin], log_c = tab[2 * bin + 1], rest = tab[2 * kLogBins + bin];
#endif
    const double ratio = z * inv, left = fma(z, inv, -ratio), lead_r = ratio - 1.0, r = lead_r + left;
    double p = fma(r, -1.0 / 8.0, 1.0 / 7.0);
    p = fma(r, p, -1.0 / 6.0);
    p = fma(r, p, 1.0 / 5.0);
    p = fma(r, p, -1.0 / 4.0);
    p = fma(r, p, 1.0 / 3.0);
    p = fma(r, p, -1.0 / 2.0);
    const double lead = fma((double)e, 0x1.62e42fefa3800p-1, log_c);   // log 2 to 42 bits behind the point
    const double sum = lead + lead_r, low = ((lead - sum) + lead_r) + left;   // lead is 0 or the larger one
    return sum + (low + fma(r * r, p, fma((double)e, 0x1.ef35793c76730p-45, rest)));
}

// The table, made once: it took 18 us of a new handle's first pass.
inline const std::array<double, 3 * kLogBins>& log_table() {
    static const std::array<double, 3 * kLogBins> table = [] {
        std::array<double, 3 * kLogBins> t;
        for (int i = 0; i < kLogBins; ++i) {
            const double c = log_value((int64_t)(kLogFrom + (i << kLogBinShift) + (1 << (kLogBinShift - 1))) << 32);
            const double inv = 1.0 / c;
            const long double log_c = -std::log((long double)inv), lead = std::nearbyint(log_c * 0x1p42L) * 0x1p-42L;
            t[2 * i] = inv;
            t[2 * i + 1] = (double)lead;
            t[2 * kLogBins + i] = (double)(log_c - lead);
        }
        return t;
    }();
    return table;
}

}  // namespace slaq
