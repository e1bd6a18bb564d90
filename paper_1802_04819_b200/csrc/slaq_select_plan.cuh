// Which way a selection takes its rows.  Host arithmetic, and compiles without CUDA.
#pragma once

#include <algorithm>

namespace slaq {

constexpr int kResidentGains = 2048;                  // gains per block up to which the whole table is predicted at once
constexpr int kBoundedRows = 60000;                   // see select_bounded
constexpr int kSampleLeast = 32, kSampleShare = 64;   // rows a block samples (predict_to_bound): at least, and one in so many

// Cores per row that enter the first histogram.
inline int select_depth(long long J, int cap, long long want, int sm_count) {
    if (J * cap <= (long long)kResidentGains * sm_count) return cap;
    const long long average = (want + J - 1) / J + 1;
    return (int)std::min<long long>(cap, std::max<long long>(16, (4 * average + 15) / 16 * 16));
}

// Whether rows are predicted down to a bound from a sample (predict_to_bound) instead of `depth` gains each.  The sample is predicted to the
// rows' ends, behind a barrier of its own, so it has to be small beside the first gains of all rows: those are at least two and a half times the
// gains of 32 rows per block.  Rows alone were the rule once; of 820 launches of 60,000 to 500,000 rows of 24 to 128 (all jobs in training,
// a third, a tenth, a hundredth of them; 0.1 to 32 cores per job) 35 were then more than 5 % slower than first gains for all (60,000 rows
// of 128: 27 -> 32 us), 13 are now, by at most 2 us; all together take 0.84 of the time.  Launch of 33,000 rows: 34 -> 37 us, of 100,000 of 64 55 -> 46, of
// 1,000,000 of 128 437 -> 201.  A sample that misleads costs the table once more (100,000 rows of 256, 32 cores per job, one job in a
// hundred in training: 225 -> 327 us).
inline bool select_bounded(long long J, int cap, long long want, int sm_count, int blocks) {
    const int depth = select_depth(J, cap, want, sm_count);
    return depth < cap && J >= kBoundedRows && 2 * J * depth >= 5LL * kSampleLeast * blocks * cap;
}

}  // namespace slaq
