// How a launch of the fit kernel is cut: warps per block, lanes per job, length classes.  Host arithmetic, and compiles without CUDA.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>

namespace slaq {

constexpr int kParked = 12;           // doubles per job and family kept in shared memory between sweeps
constexpr int kMaxFitClasses = 8;     // window-length classes of a launch
constexpr size_t kSmemLimit = 226 * 1024;   // shared memory one block may use on sm_100, less the static part

// Warps of the fit kernel's block and shared memory of each.  Fewer warps have larger slices, so that a job needs fewer lanes, and more
// registers: 128 a thread at sixteen warps, 147 to 168 at twelve (of 168), 168 to 192 at eight (of 255), where two rows overlap.  Warm
// starts spill at sixteen (104 bytes) and at twelve with several classes (200 bytes), cold fits nowhere.
enum { kSixteen, kTwelve, kEight };
constexpr int kFitWarps[3] = {16, 12, 8};
constexpr size_t kDefaultFitSlice = 13824;
constexpr size_t kFitSlices[3] = {kDefaultFitSlice, 18432, 27648};

// Window-length classes, longest first: class c holds the jobs with h_lo[c] < H <= h_hi[c] and
// gives each of them L[c] lanes.  All classes are served by one launch from one work queue
// whose slots are numbered class by class, so the longest windows start first.
struct FitClasses {
    int n;
    int h_lo[kMaxFitClasses], h_hi[kMaxFitClasses], L[kMaxFitClasses];
    int h_max;       // longest window
    int slice;       // doubles of shared memory per warp: parked sums, window rows, one spare row
};

// Doubles of shared memory per warp: the parked sums, the window rows and one spare row.  It grows if the longest window
// does not fit at 32 lanes.
inline int fit_slice(int max_hist, size_t bytes) {
    return std::max((int)(bytes / sizeof(double)), kParked * 2 + ((max_hist + 31) / 32 + 1) * 32);
}
inline int rows_at(int slice, int L) { return (slice - kParked * (64 / L)) / 32 - 1; }

struct FitPlan {
    int kind, lanes;   // index into kFitWarps; least lanes
    size_t slice_bytes;
};

// The warps of a block and the fewest lanes a job gets, from the cluster's jobs and the longest window alone.  Fewer lanes are less
// work - the solver's step and the reductions of a trial cost a warp the same whatever it carries - and longer chains of rows.  Fewer
// warps have room for fewer lanes, and leave issue slots empty.  Costs in cycles per trial: a warp alone takes `chain` + `chain_row` per row, a
// sub-partition issues `issue` + `issue_row` per row for each of its warps, of which a part counts `part` more; slots beyond what is
// resident are another wave, of which `mixed` is hidden behind the one before.  Every window is taken for full, and a fifth of the jobs,
// half the time, for new ones of a few points.
//
// A few slots more than whole waves are hidden altogether behind two waves and more, whose fits end at different trials, but not behind
// one: 19,000 full windows of 32 are four slots more than eight warps hold, and took 146 us instead of 106.
//
// Measured on 2,868 fits of 600 to 500,000 windows of up to 8 to 1,000 points (ragged, full, a fifth of them new; cold and warm) at 8, 12 and
// 16 warps and 2 to 32 lanes each: 3.5 % from the best choice on average, where sixteen warps for all with the lanes they have
// room for, the rule before, are 17.6 % from it.  Yet 81 of the fits are more than 3 % slower than those (30 more than 10 %): which last wave
// is nearly empty depends on how many windows are full, which is not known here.  Constants fitted to these fits, and sixteen warps at more
// lanes, made it 35 there and hardly fewer on 1,926 others.  No committed program repeats the sweep.
inline FitPlan fit_plan(int max_hist, long long cluster_jobs, int sm_count, size_t slice_bytes) {
    constexpr struct {
        double chain, chain_row, issue, issue_row, part, mixed;
    } cost_of[3] = {{4600, 315, 1230, 95, 0.5, 0.55}, {3600, 220, 1250, 97, 0.9, 0.4}, {3300, 190, 1340, 106, 0.1, 0.4}};
    const double jobs = (double)std::max(1LL, cluster_jobs), sub = 4.0 * sm_count;
    const bool by_size = slice_bytes == kDefaultFitSlice;
    FitPlan best = {kTwelve, 32, by_size ? kFitSlices[kTwelve] : slice_bytes};
    double least = -1.0;
    for (int L = 32; L >= 2; L >>= 1) {
        for (int kind : {kTwelve, kEight, kSixteen}) {
            const size_t bytes = by_size ? kFitSlices[kind] : slice_bytes;
            const int slice = fit_slice(max_hist, bytes);
            if (rows_at(slice, L) * L < max_hist) continue;
            if (kind == kSixteen && L > 2) continue;   // more lanes are mostly better off with more registers
            // a slice that the caller gave: as many warps as have room for it
            if (!by_size && (kind == kEight || (kind == kSixteen && sizeof(double) * ((size_t)max_hist + 16 * (size_t)slice) > kSmemLimit))) continue;
            const auto& c = cost_of[kind];
            const double rows = (max_hist + L - 1) / L, chain = c.chain + c.chain_row * rows, each = c.issue + c.issue_row * rows;
            const double resident = kFitWarps[kind] / 4;
            auto wave = [&](double n) { return std::max(chain, std::min(std::ceil(n), n + c.part) * each); };
            auto cycles = [&](double n) {   // n slots per sub-partition
                const double full = std::floor(n / resident), rest = n - full * resident;
                const double stepped = (full > 0.0 ? full * wave(resident) : 0.0) + (rest > (full < 2.0 ? 0.0 : 0.02) ? wave(rest) : 0.0);
                return c.mixed * n * std::max(each, chain / resident) + (1.0 - c.mixed) * stepped;
            };
            const double slots = jobs * L / 32.0 / sub, cost = cycles(slots) + cycles(0.8 * slots);
            if (least < 0.0 || cost <= least) best = {kind, L, bytes}, least = cost;
        }
    }
    // Beyond a wave and a half more lanes only add work, although the longest windows then get more lanes than the others.
    if (best.kind == kTwelve)
        while (best.lanes > 2 && jobs * (best.lanes / 2) >= 1.5 * 32.0 * kFitWarps[kTwelve] * sm_count) best.lanes >>= 1;
    return best;
}

// Length classes, longest first.  A warp's slice holds the parked sums of its jobs (kParked doubles per job and
// family), the window rows of 32 points and one spare row.  The class with L = 32, 16, .. lanes per job takes
// the windows that do not fit at L/2 lanes; the last one has the fewest lanes and takes the rest.
inline FitClasses fit_classes(int max_hist, const FitPlan& plan) {
    FitClasses cls = {};
    cls.h_max = max_hist;
    cls.slice = fit_slice(max_hist, plan.slice_bytes);
    int h_hi = max_hist;
    for (int L = 32; L >= plan.lanes && h_hi > 0; L >>= 1) {
        const int h_lo = L > plan.lanes ? std::max(rows_at(cls.slice, L / 2), 0) * (L / 2) : 0;
        if (h_lo >= h_hi) continue;
        cls.h_lo[cls.n] = h_lo;
        cls.h_hi[cls.n] = h_hi;
        cls.L[cls.n] = L;
        ++cls.n;
        h_hi = h_lo;
    }
    for (int c = cls.n; c < kMaxFitClasses; ++c) cls.h_lo[c] = cls.h_hi[c] = 0, cls.L[c] = 32;
    return cls;
}

}  // namespace slaq
