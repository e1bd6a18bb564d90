// From fitted curves (or a table of gains) to the allocation in one cooperative launch.
//
// The paper starts every job at one core and then gives one core at a time to the job whose next core has the
// largest predicted gain ("Scheduling Based on Quality Improvements").  Gain rows are non-increasing in n, so that
// loop hands out exactly the `want` largest gains beyond the floor, and among equal gains it serves (job id
// ascending, n ascending).  The 64-bit patterns of the gains (all >= +0) order like their values, and the threshold
// is searched on them:
//
//   A  every block predicts (or reads) the gains of its own contiguous range of jobs and counts them in a histogram
//      of 2048 bins: 64 per power of two from 2^-31 to 2, what lies below in bin 0, above in the last one.
//      -- one grid barrier --
//      Every block finds the bin of the want-th largest gain: the interval [lo, hi) the threshold lies in.
//   B  every thread walks a row from its first core: gains >= hi are handed out, the row's gains inside [lo, hi) are
//      its candidates.  A row without candidates is finished here.
//   C  the last block to arrive ranks the candidates (normally a few hundred at most: a bin is 1.6 % wide) by (gain
//      descending, job id, n) and completes their rows.  Only when there are more than kFinal of them do all blocks stay
//      and narrow the interval by another 2048 bins at a time first; candidates that are all equal are handed out
//      in job order with a prefix sum over the blocks.
//
// Tables of up to a few thousand gains take a launch of one block instead (select_small_kernel).
//
// What bounds it: for up to a few thousand jobs the latency of its steps.  It replaces eleven launches (gain kernel,
// six digits of a radix select over the whole table, counts, prefix sum, allocation) that took 90 to 110 us at every
// size up to 33,000 jobs.
//
// How much of a row is looked at.  Jobs get few cores on average, so of a large table only the first `depth` cores
// of each row enter the histogram; their bin bounds the threshold from below, and only the rows whose last gain
// still reaches that bound are continued (once, until they fall below it) before the interval is taken again.  Gains
// behind a row's first gain below the bound are below it too and can never be handed out.  Of large tables
// (select_bounded) the bound comes from a sample of the rows, before any other is looked at (predict_to_bound).
#include <math_constants.h>

#include <algorithm>
#include <cstddef>

#include "slaq_gain_curve.cuh"
#include "slaq_internal.cuh"
#include "slaq_select_plan.cuh"

namespace slaq {

namespace {

using namespace gaincurve;
using u64 = unsigned long long;

constexpr int kThreads = 1024;                       // one block per SM: half the arrivals and histogram flushes of two
constexpr int kWarps = kThreads / 32;
constexpr int kSubBits = 6;                          // bins per power of two: 64 (twice as many: the flush of 148 blocks
                                                     // costs more than the candidates it saves)
constexpr int kSub = 1 << kSubBits;
constexpr int kFine = kSelectFineBins;               // 32 powers of two
constexpr long long kBinBase = (long long)(1023 - 31) << kSubBits;
constexpr int kBinShift = 52 - kSubBits;
constexpr int kNarrowBins = kRadixBins;              // a narrowing step divides the interval by this
constexpr int kFinal = kSelectCandidates;            // candidates one block ranks
constexpr int kRankDirect = 256;                     // ranked against each other; more are narrowed in the block first
constexpr int kShortWalk = 16;                       // gains of a row its own thread walks; its warp continues
constexpr int kListWalk = 64;                        // the same where most rows are long
constexpr u64 kTopKey = 1ull << 63;                  // above every key
constexpr int kSpinLimit = 1 << 22;                  // polls of a barrier before it gives up (seconds)

__device__ __forceinline__ int fine_bin(u64 key) {
    const long long v = (long long)(key >> kBinShift) - kBinBase;
    return v < 0 ? 0 : (v > kFine - 1 ? kFine - 1 : (int)v);
}
__device__ __forceinline__ u64 bin_edge(int b) {     // smallest key of bin b; b = kFine: above every key
    return b <= 0 ? 0ull : (b >= kFine ? kTopKey : (u64)(b + kBinBase) << kBinShift);
}
__device__ __forceinline__ u64 key_of(double g) { return (u64)__double_as_longlong(g); }

// The interval the threshold lies in, the same in every block.
struct Interval {
    u64 lo, hi;      // keys >= hi are handed out, [lo, hi) are candidates
    u64 want;        // candidates still to hand out
    u64 n;           // candidates in all rows
};

struct Shared {
    union {
        unsigned int hist[kFine];
        struct {
            u64 key[kFinal], pos[kFinal];
        } cand;
    };
    unsigned int narrow[kNarrowBins];
    unsigned short idx[kFinal];
    unsigned char taken[kFinal];
    Interval iv;
    u64 scan[kWarps + 1];
    int count, n_more, flag;
    unsigned int handed[kMaxGroup][2];   // per handle: cores of the rows with candidates, candidates taken at the threshold
};

// Every block arrives; returns false (in every thread) if the others did not within the limit.
__device__ bool grid_barrier(unsigned int* bar, unsigned int target, int* flag, int32_t* err_word) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        int polls = 0;
        unsigned int seen;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
        } while (seen < target && ++polls < kSpinLimit);
        *flag = seen >= target;
        if (seen < target && err_word) atomicOr(err_word, kErrBarrier);
        __threadfence();
    }
    __syncthreads();
    return *flag != 0;
}

__device__ __forceinline__ u64 warp_inclusive(u64 v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 up = __shfl_up_sync(kFull, v, o);
        if (lane >= o) v += up;
    }
    return v;
}

// Exclusive prefix over the block's threads; every thread gets its own and *total.
__device__ u64 block_exclusive(u64 v, Shared& sh, u64* total) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const u64 incl = warp_inclusive(v);
    if (lane == 31) sh.scan[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const u64 w = lane < kWarps ? sh.scan[lane] : 0;
        const u64 s = warp_inclusive(w);
        if (lane < kWarps) sh.scan[lane] = s - w;
        if (lane == kWarps - 1) sh.scan[kWarps] = s;
    }
    __syncthreads();
    *total = sh.scan[kWarps];
    const u64 out = sh.scan[warp] + incl - v;
    __syncthreads();
    return out;
}

// The bin of the want-th largest gain from the global histogram: every warp reads one octave, and the one whose octave it is finds
// the bin.  One round trip to global memory (octave totals of their own, read first, make it two).  Fewer gains than
// wanted: an interval below everything counted, n = 0.
// kOf: which of fine (1), fine_more (2) and fine_rest (4) are added up.  What is read here is complete: every block flushed it before the
// grid barrier in front of the call, and no block adds to it behind that barrier.
template <int kOf>
__device__ void pick_first(const SelectGlobal* gl, u64 want, Shared& sh) {
    static_assert(kSub == 64 && kFine == kWarps * kSub, "a warp per octave, two bins per lane");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int top = warp * kSub + kSub - 1 - 2 * lane;   // from the octave's last bin down
    u64 v[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        v[k] = 0;
        if (kOf & 1) v[k] += __ldcg(&gl->fine[top - k]);
        if (kOf & 2) v[k] += __ldcg(&gl->fine_more[top - k]);
        if (kOf & 4) v[k] += __ldcg(&gl->fine_rest[top - k]);
    }
    const u64 sum = v[0] + v[1], incl = warp_inclusive(sum);
    if (lane == 31) sh.scan[warp] = incl;
    __syncthreads();
    const u64 octave = sh.scan[31 - lane], above = warp_inclusive(octave);
    const unsigned hit = __ballot_sync(kFull, above >= want);
    if (!hit) {
        if (threadIdx.x == 0) sh.iv = Interval{0, 0, want, 0};
    } else if (warp == 32 - __ffs(hit)) {
        const u64 before = __shfl_sync(kFull, above - octave, 31 - warp);
        const int at = __ffs(__ballot_sync(kFull, before + incl >= want)) - 1;
        if (lane == at) {
            const u64 run = before + incl - sum;
            const bool second = run + v[0] < want;
            const int b = second ? top - 1 : top;
            sh.iv = Interval{bin_edge(b), bin_edge(b + 1), want - run - (second ? v[0] : 0), second ? v[1] : v[0]};
        }
    }
}

__device__ __forceinline__ int narrow_shift(const Interval& iv) {
    const u64 width = iv.hi - iv.lo;
    const int bits = 64 - __clzll((long long)(width - 1));
    return bits > kRadixBits ? bits - kRadixBits : 0;
}

// The bin of a narrowing step's histogram (counts(b), b = 0..2047) that holds the iv.want-th largest candidate.
template <class Counts>
__device__ void pick_narrow(Counts counts, Shared& sh) {
    constexpr int per = kNarrowBins / kThreads;
    const Interval iv = sh.iv;
    const int shift = narrow_shift(iv);
    u64 v[per], sum = 0;
#pragma unroll
    for (int k = 0; k < per; ++k) sum += v[k] = counts(kNarrowBins - 1 - ((int)threadIdx.x * per + k));
    u64 total;
    u64 run = block_exclusive(sum, sh, &total);
    if (run < iv.want && iv.want <= run + sum) {
        int k = 0;
        while (k < per - 1 && run + v[k] < iv.want) run += v[k++];
        const int b = kNarrowBins - 1 - ((int)threadIdx.x * per + k);
        const u64 lo = iv.lo + ((u64)b << shift);
        sh.iv = Interval{lo, min(lo + (1ull << shift), iv.hi), iv.want - run, v[k]};
    }
    __syncthreads();
}

// Adds a block's shared counts to global ones.
__device__ void flush_first(Shared& sh, u64* fine) {
    for (int b = threadIdx.x; b < kFine; b += kThreads) {
        const unsigned int v = sh.hist[b];
        if (v) atomicAdd(&fine[b], (u64)v);
    }
}

// One row's share of the histogram: gains that fall into bin 0 (zero, or below 2^-31) are counted in a register.
__device__ __forceinline__ void count_gain(double g, bool counted, Shared& sh, unsigned int& low, int32_t* err_word) {
    if (!counted) return;
    const int b = fine_bin(key_of(g));
    if (b == 0) ++low;
    else if (index_ok(b, kFine, kErrBin, err_word)) atomicAdd(&sh.hist[b], 1u);
}

// A tile's curves in shared memory, one column per row.
struct CurveTile {
    double* v;       // [7][kThreads]
    int* kind;       // [kThreads]; -1: inactive
    __device__ void put(int r, const Curve& c, bool active) {
        v[0 * kThreads + r] = c.p0;
        v[1 * kThreads + r] = c.p1;
        v[2 * kThreads + r] = c.p2;
        v[3 * kThreads + r] = c.inv_span;
        v[4 * kThreads + r] = c.s;
        v[5 * kThreads + r] = c.w;
        v[6 * kThreads + r] = c.step_scale;
        kind[r] = active ? c.kind : -1;
    }
    __device__ Curve get(int r, double T) const {
        Curve c;
        c.kind = kind[r];
        c.p0 = v[0 * kThreads + r];
        c.p1 = v[1 * kThreads + r];
        c.p2 = v[2 * kThreads + r];
        c.inv_span = v[3 * kThreads + r];
        c.s = v[4 * kThreads + r];
        c.w = v[5 * kThreads + r];
        c.step_scale = v[6 * kThreads + r];
        c.T = T;
        return c;
    }
};

// Running minimum over the W lanes of a row (W a power of two, lanes aligned), continuing `carry`.  Most rows fall
// already, which one look at the left neighbour shows.
__device__ __forceinline__ double running_min(double g, double carry, int w, int W) {
    double left = __shfl_up_sync(kFull, g, 1, W);
    if (w == 0) left = carry;
    if (__any_sync(kFull, g > left)) {
        for (int o = 1; o < W; o <<= 1) {
            const double up = __shfl_up_sync(kFull, g, o, W);
            if (w >= o) g = fmin(g, up);
        }
        g = fmin(g, carry);
    }
    return g;
}

}  // namespace

struct SelectArgs {
    JobArrays job;
    FitArrays fit;
    const int32_t* count;    // active rows (count > 0); null: every row is active
    double* gain;            // [J][cap]
    int J, cap, first_unit;
    int depth;               // cores per row that enter the first histogram
    int W;                   // lanes per row (power of two)
    int rows;                // rows per block
    int stride;              // resident rows in shared memory: entries per row (0: rows stay in global memory)
    int keep_last;           // rows in global memory: the last of each row's first gains is kept in shared memory
    double T;
    long long want;
    SelectGlobal* gl;
    SelectState* sel;
    long long* counters;
    int32_t *gt, *eq;
    int32_t* list;           // [J], for rows with gains at or above the bound (see predict_to_bound)
    int32_t *alloc, *last_alloc, *out_alloc;
    double* reduction;
    int32_t* err_word;
    GainBasis basis;         // where the curves of unfinished rows are kept (note null: nobody asks for rows)
    // after the last row: what the next epoch finds cleared, the published statistics, and the host's mailbox
    void* zero;
    int zero_words;
    long long* published;
    Mailbox* mail;
    int32_t* mail_alloc;
    uint32_t seq;
    long long* stamps;       // [2], [3]: when the launch started and ended
};

// One handle's jobs, or those of several handles on this GPU that share one cluster's cores: each owns a run of blocks, in
// order, and all count into the first one's SelectGlobal.
constexpr int kMaxShards = kMaxGroup;
struct OneHandle {
    SelectArgs a;
    __device__ __forceinline__ int shards() const { return 1; }
    __device__ __forceinline__ const SelectArgs& of(int) const { return a; }
    __device__ __forceinline__ int mine(int* block) const {
        *block = blockIdx.x;
        return 0;
    }
};
struct ManyHandles {
    SelectArgs a[kMaxShards];
    int first_block[kMaxShards + 1];
    int n;
    __device__ __forceinline__ int shards() const { return n; }
    __device__ __forceinline__ const SelectArgs& of(int s) const { return a[s]; }
    __device__ __forceinline__ int mine(int* block) const {
        int s = 0;
        while (s + 1 < n && (int)blockIdx.x >= first_block[s + 1]) ++s;
        *block = blockIdx.x - first_block[s];
        return s;
    }
};

namespace {

__device__ __forceinline__ void store_alloc(const SelectArgs& a, int j, int cores, double R, bool active) {
    a.alloc[j] = cores;
    if (a.out_alloc) a.out_alloc[j] = cores;
    if (active && a.last_alloc) a.last_alloc[j] = cores;
    a.reduction[j] = R;
}

// The block's share of the allocation goes to the host in whole lines: written row by row as the walk ends them, 20,000
// entries were 20,000 transfers and the fence behind them took 12 to 20 us.  Every thread's stores lie before a block barrier.
__device__ __forceinline__ void mail_rows(const SelectArgs& a, int j0, int j1) {
    if (a.mail_alloc)
        for (int j = j0 + threadIdx.x; j < j1; j += kThreads) a.mail_alloc[j] = a.alloc[j];
}

// Whether the launch leaves rows unfinished: written at its end, behind the report to the host, which does not wait for it.
template <bool kCurves>
__device__ __forceinline__ void note_rows(const SelectArgs& a) {
    if (a.basis.note) *a.basis.note = GainNote{kCurves && a.depth < a.cap ? 1 : 0, a.cap, a.T};
}

// A row's candidates, entries s .. s+c-1, for the block that ranks them.  The first of them carries the row's count.
__device__ __forceinline__ void list_candidates(const SelectArgs& a, int shard, int j, int s, int c, const double* row) {
    const int at = (int)atomicAdd(&a.gl->n_cand, (unsigned int)c);
    for (int k = 0; k < c && at + k < kFinal; ++k) {
        a.gl->cand_key[at + k] = key_of(row[s + k]);
        a.gl->cand_pos[at + k] = ((u64)(k == 0 ? c : 0) << 48) | ((u64)shard << 41) | ((u64)j << 10) | (u64)(s + k);
    }
}

constexpr u64 kPosMask = (1ull << 48) - 1;

// Up to 32 candidates, a lane for each.
template <class Args>
__device__ void rank_in_a_warp(const Args& args, u64 want, int n) {
    const int lane = threadIdx.x;
    const SelectGlobal* const gl = args.of(0).gl;
    const bool has = lane < n;
    const u64 key = has ? __ldcg(&gl->cand_key[lane]) : 0, pos = has ? __ldcg(&gl->cand_pos[lane]) : 0;
    const int shard = (int)((pos >> 41) & 31), c = (int)(pos >> 48);   // c > 0: the first candidate of its row
    const int j = (int)((pos >> 10) & 0x7fffffff), s = (int)(pos & 1023);
    const SelectArgs& a = args.of(has ? shard : 0);
    double R = c > 0 ? __ldcg(&a.reduction[j]) : 0.0;
    unsigned int rank = 0;
    for (int k = 0; k < n; ++k) {
        const u64 other = __shfl_sync(kFull, key, k), other_pos = __shfl_sync(kFull, pos, k) & kPosMask;
        rank += (other > key || (other == key && other_pos < (pos & kPosMask))) ? 1 : 0;
    }
    const unsigned taken = __ballot_sync(kFull, has && rank < want), last = __ballot_sync(kFull, has && rank + 1 == want);
    const u64 tau = last ? __shfl_sync(kFull, key, __ffs(last) - 1) : 0;
    const int t = c > 0 ? __popc(taken >> lane & (c >= 32 ? kFull : (1u << c) - 1u)) : 0;   // the taken ones of a row are its first
    const int most = (int)__reduce_max_sync(kFull, (unsigned)t);
    for (int k = 0; k < most; ++k) {
        const u64 next = __shfl_sync(kFull, key, (lane + k) & 31);
        if (k < t) R += __longlong_as_double((long long)next);
    }
    if (c > 0) {
        store_alloc(a, j, s + t, R, true);
        if (a.mail_alloc) a.mail_alloc[j] = s + t;
    }
    if (lane == 0) args.of(0).sel->prefix = tau;
    for (int q = 0; q < args.shards(); ++q) {
        const unsigned cores = __reduce_add_sync(kFull, c > 0 && shard == q ? (unsigned)(s + t) : 0u);
        const unsigned ties = __ballot_sync(kFull, (taken >> lane & 1u) && key == tau && shard == q);
        if (lane == 0) {
            atomicAdd((u64*)&args.of(q).counters[6], (u64)cores);
            args.of(q).counters[7] = __popc(ties);
        }
    }
}

// The last block: hand out `iv.want` of the n <= kFinal candidates, best first, and complete their rows.
template <class Args>
__device__ void finish_candidates(const Args& args, Shared& sh) {
    const int tid = threadIdx.x;
    const SelectGlobal* const gl = args.of(0).gl;
    const int all = min((int)__ldcg(&gl->n_cand), kFinal);
    if (all <= 32) {   // one warp, without the block's barriers
        if (tid < 32) rank_in_a_warp(args, sh.iv.want, all);
        return;
    }
    if (tid < 2 * kMaxShards) sh.handed[tid >> 1][tid & 1] = 0;
    for (int i = tid; i < all; i += kThreads) {
        sh.cand.key[i] = __ldcg(&gl->cand_key[i]);
        sh.cand.pos[i] = __ldcg(&gl->cand_pos[i]);
        sh.idx[i] = (unsigned short)i;
        sh.taken[i] = 0;
    }
    int n = all;
    __syncthreads();
    while (n > kRankDirect && sh.iv.hi - sh.iv.lo > 1) {
        const int shift = narrow_shift(sh.iv);
        const u64 lo = sh.iv.lo;
        for (int b = tid; b < kNarrowBins; b += kThreads) sh.narrow[b] = 0;
        if (tid == 0) sh.count = 0;
        __syncthreads();
        int mine[kFinal / kThreads];
#pragma unroll
        for (int m = 0; m < kFinal / kThreads; ++m) {
            const int i = tid + m * kThreads;
            mine[m] = i < n ? sh.idx[i] : -1;
            if (i < n) atomicAdd(&sh.narrow[(sh.cand.key[mine[m]] - lo) >> shift], 1u);
        }
        __syncthreads();
        pick_narrow([&](int b) { return (u64)sh.narrow[b]; }, sh);
        const u64 lo2 = sh.iv.lo, hi2 = sh.iv.hi;
#pragma unroll
        for (int m = 0; m < kFinal / kThreads; ++m) {
            if (mine[m] < 0) continue;
            const u64 key = sh.cand.key[mine[m]];
            if (key >= hi2) sh.taken[mine[m]] = 1;
            else if (key >= lo2) sh.idx[atomicAdd(&sh.count, 1)] = (unsigned short)mine[m];
        }
        __syncthreads();
        n = sh.count;
        __syncthreads();
    }
    // what is left is ranked outright: 2^k threads share a candidate's comparisons
    const u64 want = sh.iv.want;
    if (tid == 0) sh.scan[0] = 0;
    for (int i = tid; i < n; i += kThreads) sh.narrow[i] = 0;
    __syncthreads();
    int share = 1;
    while (share < 32 && 2 * share * n <= kThreads) share <<= 1;
    for (int i = tid / share; i < n; i += kThreads / share) {
        const int e = sh.idx[i];
        const u64 key = sh.cand.key[e], pos = sh.cand.pos[e] & kPosMask;
        unsigned int rank = 0;
#pragma unroll 4
        for (int k = tid & (share - 1); k < n; k += share) {
            const int f = sh.idx[k];
            const u64 other = sh.cand.key[f], other_pos = sh.cand.pos[f] & kPosMask;
            rank += (other > key || (other == key && other_pos < pos)) ? 1 : 0;
        }
        if (rank) atomicAdd(&sh.narrow[i], rank);
    }
    __syncthreads();
    for (int i = tid; i < n; i += kThreads) {
        const u64 rank = sh.narrow[i];
        if (rank < want) sh.taken[sh.idx[i]] = 1;
        if (rank + 1 == want) sh.scan[0] = sh.cand.key[sh.idx[i]];
    }
    __syncthreads();
    const u64 tau = sh.scan[0];
    for (int base = 0; base < all; base += kThreads) {   // uniform trip count: the totals are added up by warps
        const int i = base + tid;
        const u64 pos = i < all ? sh.cand.pos[i] : 0;
        const int shard = (int)((pos >> 41) & 31);
        const int c = (int)(pos >> 48);   // 0: not the first candidate of its row
        const bool tie = i < all && sh.taken[i] && sh.cand.key[i] == tau;
        unsigned int cores = 0;
        if (c > 0) {
            const SelectArgs& a = args.of(shard);
            const int j = (int)((pos >> 10) & 0x7fffffff), s = (int)(pos & 1023);
            double R = __ldcg(&a.reduction[j]);
            int t = 0;                     // the taken ones of a row are its first
            while (t < c && sh.taken[i + t]) R += __longlong_as_double((long long)sh.cand.key[i + t++]);
            store_alloc(a, j, s + t, R, true);
            if (a.mail_alloc) a.mail_alloc[j] = s + t;
            cores = (unsigned int)(s + t);
        }
        for (int q = 0; q < args.shards(); ++q) {
            const unsigned int sum = __reduce_add_sync(kFull, shard == q ? cores : 0u);
            const unsigned int ties = __popc(__ballot_sync(kFull, tie && shard == q));
            if ((tid & 31) == 0) {
                if (sum) atomicAdd(&sh.handed[q][0], sum);
                if (ties) atomicAdd(&sh.handed[q][1], ties);
            }
        }
    }
    __syncthreads();
    if (tid == 0) args.of(0).sel->prefix = tau;
    if (tid < args.shards()) {
        atomicAdd((u64*)&args.of(tid).counters[6], (u64)sh.handed[tid][0]);
        args.of(tid).counters[7] = sh.handed[tid][1];
    }
}

// All blocks: narrow the interval over the rows' candidate segments (gt, eq) until kFinal candidates are left or all
// are equal; equal ones are handed out here.  Returns whether the last block still has candidates to rank, -1 after a
// barrier that was not reached.
__device__ int narrow_on_the_grid(const SelectArgs& a, int shard, SelectState* sel, Shared& sh, int j0, int j1, unsigned int& arrived) {
    const int tid = threadIdx.x;
    for (int step = 0; sh.iv.hi - sh.iv.lo > 1 && sh.iv.n > kFinal && step < kRadixPasses; ++step) {
        const int shift = narrow_shift(sh.iv);
        const u64 lo = sh.iv.lo;
        u64* global = a.gl->narrow[step];
        for (int b = tid; b < kNarrowBins; b += kThreads) sh.narrow[b] = 0;
        __syncthreads();
        for (int j = j0 + tid; j < j1; j += kThreads) {
            const int c = a.eq[j];
            const double* row = a.gain + (size_t)j * a.cap + a.gt[j];
            for (int i = 0; i < c; ++i) {
                const u64 b = (key_of(__ldcg(row + i)) - lo) >> shift;
                if (index_ok((long long)b, kNarrowBins, kErrBin, a.err_word)) atomicAdd(&sh.narrow[b], 1u);
            }
        }
        __syncthreads();
        for (int b = tid; b < kNarrowBins; b += kThreads)
            if (sh.narrow[b]) atomicAdd(&global[b], (u64)sh.narrow[b]);
        arrived += gridDim.x;
        if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) return -1;
        pick_narrow([&](int b) { return __ldcg(&global[b]); }, sh);
        const u64 lo2 = sh.iv.lo, hi2 = sh.iv.hi;
        for (int j = j0 + tid; j < j1; j += kThreads) {
            const int c = a.eq[j], s = a.gt[j];
            if (!c) continue;
            const double* row = a.gain + (size_t)j * a.cap;
            double R = a.reduction[j];
            int i = s;
            const int end = s + c;
            while (i < end && key_of(__ldcg(row + i)) >= hi2) R += __ldcg(row + i++);
            int left = 0;
            while (i + left < end && key_of(__ldcg(row + i + left)) >= lo2) ++left;
            a.gt[j] = i;
            a.eq[j] = left;
            a.reduction[j] = R;
        }
        __syncthreads();
    }
    const bool equal = sh.iv.n > kFinal;   // and the interval holds one key only
    // rows in job order: the candidates before a row decide what it gets if all are equal, its list place otherwise
    long long mine = 0;
    for (int j = j0 + tid; j < j1; j += kThreads) mine += a.eq[j];
    u64 total;
    block_exclusive((u64)mine, sh, &total);
    u64 before = 0;
    if (equal) {
        if (tid == 0) a.gl->block_eq[blockIdx.x] = (long long)total;
        arrived += gridDim.x;
        if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) return -1;
        u64 part = 0;
        for (int b = tid; b < (int)blockIdx.x; b += kThreads) part += (u64)__ldcg(&a.gl->block_eq[b]);
        block_exclusive(part, sh, &before);
    }
    long long handed = 0, ties = 0;
    for (int base = j0; base < j1; base += kThreads) {
        const int j = base + tid;
        const int c = j < j1 ? a.eq[j] : 0;
        u64 tile;
        const u64 ahead = before + block_exclusive((u64)c, sh, &tile);
        before += tile;
        if (j >= j1 || (a.count && a.count[j] <= 0)) continue;
        const int s = a.gt[j];
        if (!equal && c) {
            list_candidates(a, shard, j, s, c, a.gain + (size_t)j * a.cap);
            continue;
        }
        const int take = ahead >= sh.iv.want ? 0 : (int)min((u64)c, sh.iv.want - ahead);
        double R = a.reduction[j];
        for (int i = 0; i < take; ++i) R += a.gain[(size_t)j * a.cap + s + i];
        store_alloc(a, j, s + take, R, true);
        handed += s + take;
        ties += take;
    }
    u64 sum;
    block_exclusive((u64)handed, sh, &sum);
    if (tid == 0 && sum) atomicAdd((u64*)&a.counters[6], sum);
    if (equal) {
        block_exclusive((u64)ties, sh, &sum);
        if (tid == 0 && sum) atomicAdd((u64*)&a.counters[7], sum);
        if (tid == 0 && blockIdx.x == 0) sel->prefix = sh.iv.lo;
    }
    return equal ? 0 : 1;
}

// A tile's rows into sh.idx: those of family II from the end, the others from the front.
__device__ __forceinline__ void place_by_kind(Shared& sh, bool in, bool expo, int n_rows) {
    const int lane = threadIdx.x & 31;
    const unsigned front = __ballot_sync(kFull, in && !expo), back = __ballot_sync(kFull, in && expo), below = (1u << lane) - 1u;
    int f = 0, b = 0;
    if (lane == 0) {
        if (front) f = atomicAdd(&sh.count, __popc(front));
        if (back) b = atomicAdd(&sh.n_more, __popc(back));
    }
    f = __shfl_sync(kFull, f, 0) + __popc(front & below);
    b = __shfl_sync(kFull, b, 0) + __popc(back & below);
    if (in) sh.idx[expo ? n_rows - 1 - b : f] = (unsigned short)threadIdx.x;
}

// Whether this is the last block to get here; it then sees what the others wrote.
__device__ bool arrive_last(const SelectArgs& a, Shared& sh) {
    __syncthreads();
    if (threadIdx.x == 0) {
        if (a.mail_alloc) __threadfence_system();   // the block's share of the allocation is on its way to the host
        else __threadfence();
        sh.flag = atomicAdd(&a.gl->ticket, 1u) == gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    return sh.flag != 0;
}

// The last block, after everything else: publish the statistics, tell the host, clear the scratch for the next epoch.
template <bool kCurves, class Args>
__device__ void finish_epoch(const Args& args) {
    const int tid = threadIdx.x;
    __syncthreads();
    const SelectArgs& first = args.of(0);
    if (tid < 32) {   // the host first; the others' statistics meanwhile
        const bool mine = tid < args.shards();
        if (mine && args.of(tid).stamps) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
            args.of(tid).stamps[3] = (long long)t;
        }
        if (first.mail) {
            const unsigned err = __reduce_or_sync(kFull, mine ? (unsigned)__ldcg(args.of(tid).err_word) : 0u);
            if (tid == 0) {
                first.mail->err = (int32_t)err;
                __threadfence_system();
                first.mail->done = first.seq;
            }
        }
    } else if (tid < 32 + 16 * args.shards()) {
        const int i = tid & 15;
        const SelectArgs& a = args.of((tid - 32) >> 4);
        if (i == 0) note_rows<kCurves>(a);
        if (a.published) a.published[i] = i == 15 ? (long long)__ldcg(&first.sel->prefix) : __ldcg(&a.counters[i]);
    }
    __syncthreads();
    for (int s = 0; s < args.shards(); ++s) {
        const SelectArgs& a = args.of(s);
        if (a.zero)
            for (int i = tid; i < a.zero_words; i += kThreads) static_cast<u64*>(a.zero)[i] = 0;
    }
}

// A block whose wait at a barrier ran out ends here (the error word says so already).  Blocks that were let through meet the next
// barrier without it and end here too, so all of them arrive, and the last one leaves the scratch as the next epoch expects it:
// nobody clears it between two epochs that are queued one behind the other.
template <bool kCurves, class Args>
__device__ void give_up(const Args& args, const SelectArgs& a, Shared& sh) {
    if (arrive_last(a, sh)) finish_epoch<kCurves>(args);
}

// A tile's curves into shared memory, and its rows into sh.idx, family II's last: the rows of a warp are then of one family, and
// only one of the two formulas is walked through (a gain costs 30 to 75 instructions of the fp64 pipe in one family, the sum in
// both).  keep: the curves are also kept for rows that are asked for later.
__device__ __forceinline__ void load_tile(const SelectArgs& a, Shared& sh, CurveTile& tile, int base, int n_rows, bool keep) {
    const int tid = threadIdx.x;
    bool expo = false;
    if (tid < n_rows) {
        const int j = base + tid;
        bool no_time = false;
        const bool active = a.count[j] > 0;
        const Curve c = load_curve(a.job, a.fit, j, a.J, a.T, &no_time);
        if (no_time) a.fit.status[j] = SLAQ_JOB_NO_TIME;
        tile.put(tid, c, active);
        if (keep) keep_curve(a.basis, j, a.J, c, active ? c.kind : 3);
        expo = active && c.kind == 1;
    }
    place_by_kind(sh, tid < n_rows, expo, n_rows);
    __syncthreads();
}

// The counts of bin 0 that threads kept in a register join the others; every thread's counts lie before the block barrier.
__device__ __forceinline__ void add_low(Shared& sh, unsigned int low) {
    low = __reduce_add_sync(kFull, low);
    if ((threadIdx.x & 31) == 0 && low) atomicAdd(&sh.hist[0], low);
    __syncthreads();
}

// Half a warp's row from gain `from` on, predicted, written and counted where the key lies in [lo, hi), until it falls below `until`.
__device__ __forceinline__ void predict_row(const SelectArgs& a, Shared& sh, bool in, int j, int from, u64 lo, u64 hi, u64 until, bool store,
                                            unsigned int& low) {
    constexpr int W = 16;
    const int w = threadIdx.x & (W - 1);
    double* const row = a.gain + (size_t)j * a.cap;
    Curve c;
    c.kind = 3;
    double carry = CUDART_INF;
    bool active = false;
    if (in) {
        bool no_time = false;
        c = load_curve<true>(a.job, a.fit, j, a.J, a.T, &no_time);
        active = a.count[j] > 0;
        if (from > 0) carry = row[from - 1];
    }
    bool on = in;
    for (int n0 = from; n0 < a.cap && __any_sync(kFull, on); n0 += W) {
        const int i = n0 + w;
        const bool has = on && i < a.cap && index_ok((long long)j * a.cap + i, (long long)a.J * a.cap, kErrGain, a.err_word);
        double g = 0.0;
        if (has) g = c.kind == 3 ? 0.0 : raw_gain(c, i + 1);
        g = running_min(g, carry, w, W);
        if (has && store) row[i] = g;
        count_gain(g, has && active && i + 1 >= a.first_unit && key_of(g) >= lo && key_of(g) < hi, sh, low, a.err_word);
        carry = __shfl_sync(kFull, g, W - 1, W);
        on = on && key_of(carry) >= until;
    }
}

// Large tables are not predicted as a whole: few jobs get more than their first core (of 1,000,000 jobs one in ten), so gains are
// predicted down to a bound that lies just below the threshold.  Where that is, a sample of the rows tells - every block takes some of its
// own, predicts them to the end and adds them to a histogram; the bound is the bin at the rank that the gains wanted have in the
// sample, and five times the deviation such a rank can have at most (sqrt(cap x rank): a row counts for up to cap) beyond.  Then every row is predicted
// four gains at a time until it falls below the bound.  Rows without a gain at or above it keep their floor and are done; the others are
// listed, those that need more than four gains from the front, and their gains make the histogram the interval is taken from.
// Should the sample have misled (fewer gains than wanted at or above the bound), every row is predicted to its end: slow, and the same result.
// Predicting the first 16 gains of every row and taking the bound from those instead continued rows for a bound far below the
// threshold, since they hold too few of the gains of the rows that get many (launch for 1,000,000 rows of 128: 437 -> 201 us, first gains
// 142 -> 60 of them, continued rows 151 -> 50, walk 106 -> 30).
// Returns false after a barrier that was not reached.
constexpr int kFirstGains = 4;
template <class Args>
__device__ bool predict_to_bound(const Args& args, const SelectArgs& a, Shared& sh, CurveTile& tile, int j0, int j1, unsigned int& arrived,
                                 bool* listed, int* n_more, int* n_some, long long* handed) {
    const int tid = threadIdx.x, lane = tid & 31, n = j1 - j0;
    const int floor_cores = a.first_unit - 1;
    int32_t* const list = a.list + j0;
    unsigned int low = 0;
    // the next two rows of n for the calling warp: a row for each half of it
    auto draw = [&](int limit, bool* in) {
        int r = lane == 0 ? (int)atomicAdd(&sh.narrow[2], 2u) : 0;
        r = __shfl_sync(kFull, r, 0) + (lane >> 4);
        *in = r < limit;
        return r;
    };
    auto reset = [&]() {   // counters and the histogram
        __syncthreads();
        for (int i = tid; i < kFine; i += kThreads) sh.hist[i] = 0;
        if (tid < 3) sh.narrow[tid] = 0;
        low = 0;
        __syncthreads();
    };
    u64 bound = ~0ull;   // nothing wanted: above every gain
    if (a.want > 0) {
        const int n_sample = min(n, max(kSampleLeast, n / kSampleShare));
        if (tid == 0) {
            sh.narrow[2] = 0;
            atomicAdd(&a.gl->sampled, (unsigned int)n_sample);
        }
        __syncthreads();
        for (;;) {
            bool in;
            const int r = draw(n_sample, &in);
            if (__all_sync(kFull, !in)) break;
            // one row of each of n_sample equal parts
            const int j = in ? j0 + (int)(((long long)r * n + (unsigned int)(r * 2654435761u + blockIdx.x * 40503u) % (unsigned int)n) / n_sample) : j0;
            predict_row(a, sh, in, j, 0, bin_edge(1), kTopKey, bin_edge(1), false, low);
        }
        __syncthreads();
        flush_first(sh, a.gl->fine);
        arrived += gridDim.x;
        if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) return false;
        long long J = 0;
        for (int q = 0; q < args.shards(); ++q) J += args.of(q).J;
        const double rank = (double)a.want * ((double)__ldcg(&a.gl->sampled) / (double)J);
        pick_first<1>(a.gl, (u64)(rank + 5.0 * sqrt((double)a.cap * rank) + 8.0), sh);
        __syncthreads();
        bound = sh.iv.lo;
    }
    reset();
    for (int base = j0; base < j1; base += kThreads) {
        const int n_rows = min(kThreads, j1 - base);
        if (tid == 0) sh.count = sh.n_more = 0;
        __syncthreads();
        load_tile(a, sh, tile, base, n_rows, true);
        const int w = tid & (kFirstGains - 1);
        for (int r0 = 0; r0 < n_rows; r0 += kThreads / kFirstGains) {   // uniform trip count: the row steps use warp shuffles
            const int at = r0 + tid / kFirstGains;
            const bool in = at < n_rows;
            const int r = in ? sh.idx[at] : 0, j = base + r;
            Curve c;
            c.kind = -1;
            if (in) c = tile.get(r, a.T);
            const bool active = c.kind >= 0;
            const bool has = in && index_ok((long long)j * a.cap + w, (long long)a.J * a.cap, kErrGain, a.err_word);
            const double g = running_min(has && active && c.kind != 3 ? raw_gain(c, w + 1) : 0.0, CUDART_INF, w, kFirstGains);
            const double first = __shfl_sync(kFull, g, floor_cores, kFirstGains), last = __shfl_sync(kFull, g, kFirstGains - 1, kFirstGains);
            const bool some = active && key_of(first) >= bound, more = some && key_of(last) >= bound;
            if (has && some) a.gain[(size_t)j * a.cap + w] = g;
            count_gain(g, has && some && w + 1 >= a.first_unit && key_of(g) >= bound, sh, low, a.err_word);
            if (in && w == 0) {   // the row's curve is in its lanes' registers: its place holds the first gain now
                tile.v[r] = g;
                sh.taken[r] = some ? (more ? 2 : 1) : 0;
            }
        }
        __syncthreads();
        if (tid < n_rows) {
            const int j = base + tid, state = sh.taken[tid];
            const bool active = tile.kind[tid] >= 0;
            if (state == 0) {
                store_alloc(a, j, active ? floor_cores : 0, active && floor_cores ? tile.v[tid] : 0.0, active);
                *handed += active ? floor_cores : 0;
            } else if (state == 2) {
                const int at = (int)atomicAdd(&sh.narrow[0], 1u);
                if (index_ok(at, n, kErrJob, a.err_word)) list[at] = j;
            } else {
                const int at = n - 1 - (int)atomicAdd(&sh.narrow[1], 1u);
                if (index_ok(at, n, kErrJob, a.err_word)) list[at] = j;
            }
        }
        __syncthreads();
    }
    *listed = true;
    *n_more = (int)sh.narrow[0];
    *n_some = (int)sh.narrow[1];
    for (;;) {
        bool in;
        const int r = draw(*n_more, &in);
        if (__all_sync(kFull, !in)) break;
        predict_row(a, sh, in, in && index_ok(r, n, kErrJob, a.err_word) ? list[r] : j0, kFirstGains, bound, kTopKey, bound, true, low);
    }
    add_low(sh, low);
    flush_first(sh, a.gl->fine_more);
    arrived += gridDim.x;
    if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) return false;
    if (a.want > 0) {
        pick_first<2>(a.gl, (u64)a.want, sh);
    } else if (tid == 0) {
        sh.iv = Interval{~0ull, ~0ull, 0, 0};
    }
    __syncthreads();
    if (sh.iv.hi > 0 || bound == 0) return true;
    // the sample has misled: all gains below the bound as well, and all rows to be walked
    reset();
    *listed = false;
    *handed = 0;
    for (;;) {
        bool in;
        const int r = draw(n, &in);
        if (__all_sync(kFull, !in)) break;
        predict_row(a, sh, in, in ? j0 + r : j0, 0, 0, bound, 0, true, low);
    }
    add_low(sh, low);
    flush_first(sh, a.gl->fine_rest);
    arrived += gridDim.x;
    if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) return false;
    pick_first<6>(a.gl, (u64)a.want, sh);
    __syncthreads();
    return true;
}

// kCurves: gains are predicted from the fitted curves and written to the table (rows beyond `depth` only as far as they
// were continued); otherwise the table is read.
// kBounded: see predict_to_bound; a kernel of its own, since the two ways in one cost the smaller tables 2 to 5 us.
template <bool kCurves, bool kBounded, class Args>
__global__ void __launch_bounds__(kThreads, 1) select_kernel(const __grid_constant__ Args args) {
    extern __shared__ double dyn[];
    __shared__ Shared sh;
    const int tid = threadIdx.x;
    int block;
    const int shard = args.mine(&block);
    const SelectArgs& a = args.of(shard);
    const int j0 = min(block * a.rows, a.J), j1 = min(j0 + a.rows, a.J);
    after_previous();
    if (block == 0 && tid == 0 && a.stamps) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        a.stamps[2] = (long long)t;
    }
    const bool resident = a.stride > 0;
    CurveTile tile;
    tile.v = dyn;
    tile.kind = reinterpret_cast<int*>(dyn + 7 * kThreads);
    double* const rows_sh = dyn + (kCurves ? 7 * kThreads + kThreads / 2 : 0);   // resident rows, or each row's last gain
    unsigned int arrived = 0;

    for (int i = tid; i < kFine; i += kThreads) sh.hist[i] = 0;
    // the counts of continued rows and the narrowing histograms, should they be needed: cleared by all blocks before the first barrier
    constexpr int kLater = (int)((offsetof(SelectGlobal, cand_key) - offsetof(SelectGlobal, fine_more)) / sizeof(u64));
    u64* const later = reinterpret_cast<u64*>(reinterpret_cast<char*>(a.gl) + offsetof(SelectGlobal, fine_more));
    for (int i = blockIdx.x * kThreads + tid; i < kLater; i += gridDim.x * kThreads) later[i] = 0;
    if (tid == 0) sh.count = sh.n_more = 0;
    __syncthreads();

    long long handed = 0;
    bool listed = false;             // B walks the rows of `list`: n_more from the front of the block's part, n_some from its end
    int n_more = 0, n_some = 0;
    const int32_t* const list = kBounded ? a.list + j0 : nullptr;
    if constexpr (kBounded) {
        if (!predict_to_bound(args, a, sh, tile, j0, j1, arrived, &listed, &n_more, &n_some, &handed)) {
            give_up<kCurves>(args, a, sh);
            return;
        }
    } else {
        // ---- A: the first `depth` gains of every row ----
        unsigned int low = 0;
        const int W = a.W, w = tid & (W - 1), groups = kThreads / W;
        for (int base = j0; base < j1; base += kThreads) {
            const int n_rows = min(kThreads, j1 - base);
            if constexpr (kCurves) load_tile(a, sh, tile, base, n_rows, a.depth < a.cap);
            for (int r0 = 0; r0 < n_rows; r0 += groups) {   // uniform trip count: the row steps use warp shuffles
                const int at = r0 + tid / W;
                const bool in = at < n_rows;
                const int r = in ? (kCurves ? sh.idx[at] : at) : 0;
                const int j = base + r;
                Curve c;
                bool active = false;
                if (kCurves) {
                    if (in) {
                        c = tile.get(r, a.T);
                        active = c.kind >= 0;
                        if (!active) c.kind = 3;
                    }
                } else if (in) {
                    active = !a.count || a.count[j] > 0;
                }
                double* const row = a.gain + (size_t)j * a.cap;
                double carry = CUDART_INF;
                for (int n0 = 0; n0 < a.depth; n0 += W) {
                    const int i = n0 + w;
                    const bool has = in && i < a.depth && index_ok((long long)j * a.cap + i, (long long)a.J * a.cap, kErrGain, a.err_word);
                    double g = 0.0;
                    if (kCurves) {
                        if (has) g = c.kind == 3 ? 0.0 : raw_gain(c, i + 1);
                        g = running_min(has ? g : 0.0, carry, w, W);
                        carry = __shfl_sync(kFull, g, W - 1, W);
                        if (has) row[i] = g;
                    } else if (has) {
                        g = row[i];
                    }
                    if (has && resident) rows_sh[(base - j0 + r) * a.stride + i] = g;
                    else if (has && a.keep_last && i == a.depth - 1) rows_sh[base - j0 + r] = g;
                    count_gain(g, has && active && i + 1 >= a.first_unit, sh, low, a.err_word);
                }
            }
            if (kCurves && tid == 0) sh.count = sh.n_more = 0;
            __syncthreads();
        }
        add_low(sh, low);
        flush_first(sh, a.gl->fine);
        arrived += gridDim.x;
        if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) {
            give_up<kCurves>(args, a, sh);
            return;
        }
        if (a.want > 0) {
            pick_first<1>(a.gl, (u64)a.want, sh);
        } else if (tid == 0) {
            sh.iv = Interval{~0ull, ~0ull, 0, 0};   // nothing wanted: a threshold above every gain
        }
        __syncthreads();

        // ---- rows that may reach the threshold beyond `depth` are continued ----
        if (a.depth < a.cap && a.want > 0) {
            const u64 bound = sh.iv.lo;
            for (int i = tid; i < kFine; i += kThreads) sh.hist[i] = 0;
            low = 0;
            for (int base = j0; base < j1; base += kThreads) {
                if (tid == 0) sh.count = sh.n_more = 0;
                __syncthreads();
                const int mine = base + tid;
                if (mine < j1 && (!a.count || a.count[mine] > 0) &&
                    key_of(a.keep_last ? rows_sh[mine - j0] : a.gain[(size_t)mine * a.cap + a.depth - 1]) >= bound) {
                    const bool expo = kCurves && a.fit.status[mine] == SLAQ_JOB_FITTED && a.fit.family[mine] == 1;   // those last, as above
                    sh.narrow[expo ? kThreads - 1 - atomicAdd(&sh.n_more, 1) : atomicAdd(&sh.count, 1)] = (unsigned int)mine;
                }
                __syncthreads();
                const int n_front = sh.count, n_all = n_front + sh.n_more;
                for (int r0 = 0; r0 < n_all; r0 += groups) {
                    const int r = r0 + tid / W;
                    const bool in = r < n_all;
                    const int j = in ? (int)sh.narrow[r < n_front ? r : kThreads - 1 - (r - n_front)] : base;
                    double* const row = a.gain + (size_t)j * a.cap;
                    Curve c;
                    c.kind = 3;
                    double carry = CUDART_INF;
                    if (kCurves && in) {
                        bool no_time = false;
                        c = load_curve(a.job, a.fit, j, a.J, a.T, &no_time);
                        carry = row[a.depth - 1];
                    }
                    bool on = in;
                    for (int n0 = a.depth; n0 < a.cap && __any_sync(kFull, on); n0 += W) {
                        const int i = n0 + w;
                        const bool has = on && i < a.cap && index_ok((long long)j * a.cap + i, (long long)a.J * a.cap, kErrGain, a.err_word);
                        double g = 0.0;
                        if (kCurves) {
                            if (has) g = c.kind == 3 ? 0.0 : raw_gain(c, i + 1);
                            g = running_min(g, carry, w, W);
                            if (has) row[i] = g;
                        } else if (has) {
                            g = row[i];
                        }
                        count_gain(g, has && i + 1 >= a.first_unit, sh, low, a.err_word);
                        carry = __shfl_sync(kFull, g, W - 1, W);
                        on = on && key_of(carry) >= bound;
                    }
                }
                __syncthreads();
            }
            add_low(sh, low);
            flush_first(sh, a.gl->fine_more);
            arrived += gridDim.x;
            if (!grid_barrier(&a.gl->barrier, arrived, &sh.flag, a.err_word)) {
                give_up<kCurves>(args, a, sh);
                return;
            }
            pick_first<3>(a.gl, (u64)a.want, sh);
            __syncthreads();
        }
    }

    // ---- B: every row that may have gains at or above the interval, up to it ----
    const Interval iv = sh.iv;
    const bool few = iv.n <= kFinal;
    const int lane = tid & 31;
    const int n_walk = listed ? n_more + n_some : j1 - j0;
    if (listed && !few) {   // the others have no candidates
        for (int j = j0 + tid; j < j1; j += kThreads) {
            a.gt[j] = a.count[j] > 0 ? a.first_unit - 1 : 0;
            a.eq[j] = 0;
        }
        __syncthreads();
    }
    // few rows per block, or long ones, are spread over its warps, one per warp at first
    const int pitch = n_walk <= (listed ? kThreads : kThreads / 4) ? kWarps : 1;
    const int slot0 = pitch == 1 ? tid & ~31 : tid >> 5, slot = slot0 + pitch * lane;
    for (int base = 0; base < n_walk; base += kThreads) {   // uniform trip count: a warp finishes its long rows together
        const int at = base + slot;
        const bool in = at < n_walk;
        const int place = at < n_more ? at : j1 - j0 - 1 - (at - n_more);   // in the list: the longer ones from its front, the others from its end
        const int j = !in ? j0 : !listed ? j0 + at : index_ok(place, j1 - j0, kErrJob, a.err_word) ? list[place] : j0;
        const bool active = in && (!a.count || a.count[j] > 0);
        const double* row = resident ? rows_sh + (size_t)(j - j0) * a.stride : a.gain + (size_t)j * a.cap;
        int s = 0, c = 0;
        double R = 0.0;
        bool more = false;
        if (active) {
            if (a.first_unit == 2) R = row[0], s = 1;
            const int end = min(a.cap, listed ? kListWalk : kShortWalk);
            more = s < a.cap;
            while (more && s < end) {
                double g[4];   // four loads in flight; entries behind a row's first gain below the interval mean nothing
#pragma unroll
                for (int k = 0; k < 4; ++k) g[k] = s + k < end ? row[s + k] : 0.0;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (more && s < end) {
                        if (key_of(g[k]) >= iv.hi) R += g[k], ++s;
                        else more = false;
                    }
                }
            }
            more = more && s < a.cap;   // every gain so far is handed out
        }
        for (unsigned todo = __ballot_sync(kFull, more); todo; todo &= todo - 1) {
            const int r = __ffs(todo) - 1;
            const int jr = __shfl_sync(kFull, j, r);
            const double* far = resident ? rows_sh + (size_t)(jr - j0) * a.stride : a.gain + (size_t)jr * a.cap;
            int at_n = __shfl_sync(kFull, s, r);
            double sum = __shfl_sync(kFull, R, r);
            for (bool on = true; on && at_n < a.cap;) {
                const double g = at_n + lane < a.cap ? far[at_n + lane] : 0.0;
                const unsigned stop = __ballot_sync(kFull, at_n + lane >= a.cap || key_of(g) < iv.hi);
                const int n = stop ? __ffs(stop) - 1 : 32;
                for (int k = 0; k < n; ++k) sum += __shfl_sync(kFull, g, k);   // in order, as the row's own thread adds
                at_n += n;
                on = n == 32;
            }
            if (lane == r) s = at_n, R = sum;
        }
        if (!in) continue;
        if (active)
            while (s + c < a.cap && key_of(row[s + c]) >= iv.lo) ++c;
        if (few && c == 0) {
            store_alloc(a, j, s, R, active);
            handed += s;
        } else {
            a.reduction[j] = R;
            if (few) {
                list_candidates(a, shard, j, s, c, row);
            } else {
                a.gt[j] = s;
                a.eq[j] = c;
                if (!active) store_alloc(a, j, 0, 0.0, false);
            }
        }
    }
    if (few) {
        u64 sum;
        block_exclusive((u64)handed, sh, &sum);
        if (tid == 0 && sum) atomicAdd((u64*)&a.counters[6], sum);
        mail_rows(a, j0, j1);
    } else {
        __syncthreads();
        const int next = narrow_on_the_grid(a, shard, args.of(0).sel, sh, j0, j1, arrived);
        if (next < 0) {
            give_up<kCurves>(args, a, sh);
            return;
        }
        mail_rows(a, j0, j1);   // rows with candidates that are still to be ranked are written again after that
        if (next == 0) {
            if (arrive_last(a, sh)) finish_epoch<kCurves>(args);
            return;
        }
    }

    // ---- C: the last block to get here ranks the candidates ----
    if (!arrive_last(a, sh)) return;
    if (sh.iv.n > 0) finish_candidates(args, sh);
    else if (tid == 0) args.of(0).sel->prefix = ~0ull;
    finish_epoch<kCurves>(args);
}

// Few gains: one block does everything in shared memory, with no grid barrier and nothing but results in global memory.
// The launch above takes 13 us for any small table, most of it round trips to global memory: flushing and
// reading the histogram, arriving at two counters, listing and reading candidates.  This one takes 4.8 us for 128
// gains, 7.3 for 2,048 and 10.5 for 160 rows of 32: one SM predicts about a thousand gains per microsecond, so the two
// meet near 6,000.
template <bool kCurves>
__global__ void __launch_bounds__(kThreads, 1) select_small_kernel(const __grid_constant__ OneHandle args) {
    extern __shared__ double dyn[];
    __shared__ Shared sh;
    const SelectArgs& a = args.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    CurveTile tile;
    tile.v = dyn;
    tile.kind = reinterpret_cast<int*>(dyn + 7 * kThreads);
    double* const rows = dyn + (kCurves ? 7 * kThreads + kThreads / 2 : 0);

    for (int i = tid; i < kFine; i += kThreads) sh.hist[i] = 0;
    if (tid == 0) sh.count = 0;
    after_previous();
    if (a.stamps) note_time(a.stamps + 2);
    if (kCurves && tid < a.J) {
        bool no_time = false;
        const bool active = a.count[tid] > 0;
        const Curve c = load_curve<true, true>(a.job, a.fit, tid, a.J, a.T, &no_time);
        if (no_time) a.fit.status[tid] = SLAQ_JOB_NO_TIME;
        tile.put(tid, c, active);
    }
    __syncthreads();

    // ---- A: all gains, and their histogram ----
    unsigned int low = 0;
    const int W = a.W, w = tid & (W - 1), groups = kThreads / W;
    for (int r0 = 0; r0 < a.J; r0 += groups) {   // uniform trip count: the row steps use warp shuffles
        const int r = r0 + tid / W;
        const bool in = r < a.J;
        Curve c;
        c.kind = 3;
        bool active = false;
        if (in) {
            if (kCurves) {
                c = tile.get(r, a.T);
                active = c.kind >= 0;
                if (!active) c.kind = 3;
            } else {
                active = !a.count || a.count[r] > 0;
            }
        }
        double* const row = a.gain + (size_t)(in ? r : 0) * a.cap;
        double carry = CUDART_INF;
        for (int n0 = 0; n0 < a.cap; n0 += W) {
            const int i = n0 + w;
            const bool has = in && i < a.cap && index_ok((long long)r * a.cap + i, (long long)a.J * a.cap, kErrGain, a.err_word);
            double g = 0.0;
            if (kCurves) {
                if (has) g = c.kind == 3 ? 0.0 : raw_gain(c, i + 1);
                g = running_min(g, carry, w, W);
                carry = __shfl_sync(kFull, g, W - 1, W);
                if (has) row[i] = g;
            } else if (has) {
                g = row[i];
            }
            if (has) rows[r * a.stride + i] = g;
            count_gain(g, has && active && i + 1 >= a.first_unit, sh, low, a.err_word);
        }
    }
    low = __reduce_add_sync(kFull, low);
    if (lane == 0 && low) atomicAdd(&sh.hist[0], low);
    __syncthreads();
    // ---- the bin of the want-th largest gain: the octave by one warp each, then its bins ----
    const unsigned int octave = __reduce_add_sync(kFull, sh.hist[warp * kSub + lane] + sh.hist[warp * kSub + 32 + lane]);
    if (lane == 0) sh.narrow[warp] = octave;
    __syncthreads();
    if (warp == 0) {
        const u64 want = (u64)a.want;
        const u64 c = sh.narrow[31 - lane], incl = warp_inclusive(c);
        const unsigned hit = __ballot_sync(kFull, incl >= want);
        if (a.want <= 0) {
            if (lane == 0) sh.iv = Interval{~0ull, ~0ull, 0, 0};   // nothing wanted: a threshold above every gain
        } else if (!hit) {
            if (lane == 0) sh.iv = Interval{0, 0, want, 0};
        } else {
            const int at = __ffs(hit) - 1;
            const u64 above = __shfl_sync(kFull, incl - c, at);
            const int top = (31 - at) * kSub + kSub - 1 - 2 * lane;
            const u64 first = sh.hist[top], sum = first + sh.hist[top - 1];
            const u64 incl2 = warp_inclusive(sum);
            const int at2 = __ffs(__ballot_sync(kFull, above + incl2 >= want)) - 1;
            if (lane == at2) {
                const u64 run = above + incl2 - sum;
                const bool second = run + first < want;
                const int b = second ? top - 1 : top;
                sh.iv = Interval{bin_edge(b), bin_edge(b + 1), want - run - (second ? first : 0), second ? sum - first : first};
            }
        }
    }
    __syncthreads();

    // ---- B: a thread per row, rows dealt out to the warps: what lies above the interval, and the row's candidates ----
    const int j = warp + kWarps * lane;
    const bool in = j < a.J, active = in && (!a.count || a.count[j] > 0);
    const double* const row = rows + (size_t)j * a.stride;
    int s = 0, c = 0;
    double R = 0.0;
    {
        const u64 lo = sh.iv.lo, hi = sh.iv.hi;
        bool more = false;
        if (active) {
            if (a.first_unit == 2) R = row[0], s = 1;
            const int end = min(a.cap, kShortWalk);
            more = s < a.cap;
            while (more && s < end) {
                const double g = row[s];
                more = key_of(g) >= hi;
                if (more) R += g, ++s;
            }
            more = more && s < a.cap;   // every gain so far is handed out
        }
        for (unsigned todo = __ballot_sync(kFull, more); todo; todo &= todo - 1) {   // the warp continues a long row
            const int r = __ffs(todo) - 1;
            const double* const far = rows + (size_t)(warp + kWarps * r) * a.stride;
            int at = __shfl_sync(kFull, s, r);
            double sum = __shfl_sync(kFull, R, r);
            for (bool on = true; on && at < a.cap;) {
                const double g = at + lane < a.cap ? far[at + lane] : 0.0;
                const unsigned stop = __ballot_sync(kFull, at + lane >= a.cap || key_of(g) < hi);
                const int n = stop ? __ffs(stop) - 1 : 32;
                for (int k = 0; k < n; ++k) sum += __shfl_sync(kFull, g, k);   // in order, as the row's own thread adds
                at += n;
                on = n == 32;
            }
            if (lane == r) s = at, R = sum;
        }
        if (active)
            while (s + c < a.cap && key_of(row[s + c]) >= lo) ++c;
    }
    // ---- the interval is narrowed until its candidates can be ranked, or are all equal ----
    for (int step = 0; sh.iv.n > kRankDirect && sh.iv.hi - sh.iv.lo > 1 && step < kRadixPasses; ++step) {
        const int shift = narrow_shift(sh.iv);
        const u64 lo = sh.iv.lo;
        for (int b = tid; b < kNarrowBins; b += kThreads) sh.narrow[b] = 0;
        __syncthreads();
        for (int k = 0; k < c; ++k) {
            const u64 b = (key_of(row[s + k]) - lo) >> shift;
            if (index_ok((long long)b, kNarrowBins, kErrBin, a.err_word)) atomicAdd(&sh.narrow[b], 1u);
        }
        __syncthreads();
        pick_narrow([&](int b) { return (u64)sh.narrow[b]; }, sh);
        const u64 lo2 = sh.iv.lo, hi2 = sh.iv.hi;
        const int end = s + c;
        while (s < end && key_of(row[s]) >= hi2) R += row[s++];
        c = 0;
        while (s + c < end && key_of(row[s + c]) >= lo2) ++c;
    }
    __syncthreads();   // every thread has read the interval and the histogram for the last time
    // ---- C: how many of a row's candidates are handed out ----
    const u64 want = sh.iv.want, n = sh.iv.n;
    int take = 0;
    u64 tau = ~0ull;
    if (n > kRankDirect) {   // all equal: in job order
        if (in) sh.idx[j] = (unsigned short)c;
        __syncthreads();
        u64 total;
        const u64 mine = block_exclusive(tid < a.J ? sh.idx[tid] : 0, sh, &total);
        if (tid < a.J) sh.cand.pos[tid] = mine;
        __syncthreads();
        const u64 before = in ? sh.cand.pos[j] : 0;
        take = before >= want ? 0 : (int)min((u64)c, want - before);
        tau = sh.iv.lo;
    } else if (n > 0) {
        for (int i = tid; i < a.J; i += kThreads) sh.narrow[i] = 0;
        if (c) {
            const int at = atomicAdd(&sh.count, c);
            for (int k = 0; k < c; ++k) {
                sh.cand.key[at + k] = key_of(row[s + k]);
                sh.cand.pos[at + k] = ((u64)j << 10) | (u64)(s + k);
            }
        }
        __syncthreads();
        int share = kThreads / kRankDirect;   // threads per candidate
        while (share < 32 && 2 * share * (int)n <= kThreads) share <<= 1;
        const int i = tid / share;
        const bool mine = i < (int)n;
        const u64 key = mine ? sh.cand.key[i] : 0, pos = mine ? sh.cand.pos[i] : 0;
        unsigned int rank = 0;
        if (mine)
            for (int k = tid & (share - 1); k < (int)n; k += share) {
                const u64 other = sh.cand.key[k];
                rank += (other > key || (other == key && sh.cand.pos[k] < pos)) ? 1 : 0;
            }
        for (int o = share >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(kFull, rank, o);
        if (mine && (tid & (share - 1)) == 0) {
            if (rank < want) atomicAdd(&sh.narrow[(int)(pos >> 10)], 1u);   // the taken ones of a row are its first
            if (rank + 1 == want) sh.scan[0] = key;
        }
        __syncthreads();
        if (in) take = (int)sh.narrow[j];
        tau = sh.scan[0];
    }
    int ties = 0;
    for (int k = 0; k < take; ++k) {
        ties += key_of(row[s + k]) == tau;
        R += row[s + k];
    }
    if (in) {
        store_alloc(a, j, active ? s + take : 0, R, active);
        sh.idx[j] = (unsigned short)(active ? s + take : 0);
    }
    // ---- totals of the statistics, the host's mailbox, a cleared scratch for the next epoch ----
    const unsigned int cores = __reduce_add_sync(kFull, (unsigned int)(active ? s + take : 0));
    ties = __reduce_add_sync(kFull, ties);
    __syncthreads();   // and all results are stored
    if (a.mail_alloc && tid < a.J) a.mail_alloc[tid] = sh.idx[tid];   // in whole lines
    __syncthreads();
    if (lane == 0) sh.hist[2 * warp] = cores, sh.hist[2 * warp + 1] = ties;
    if (a.stamps) note_time(a.stamps + 3);
    if (tid == 0 && a.mail) {
        a.mail->err = __ldcg(a.err_word);
        __threadfence_system();
        a.mail->done = a.seq;
    }
    __syncthreads();
    if (warp == 1) {
        const unsigned int all = __reduce_add_sync(kFull, sh.hist[2 * lane]), tied = __reduce_add_sync(kFull, sh.hist[2 * lane + 1]);
        if (lane == 0) a.sel->prefix = tau;
        if (lane == 16) note_rows<kCurves>(a);
        if (lane < 16) {
            const long long v = lane == 6 ? all : lane == 7 ? tied : lane == 15 ? (long long)tau : __ldcg(&a.counters[lane]);
            if (a.published) a.published[lane] = v;
            else if (lane == 6 || lane == 7) a.counters[lane] = v;
        }
    }
    __syncthreads();
    if (a.zero)
        for (int i = tid; i < a.zero_words; i += kThreads) static_cast<u64*>(a.zero)[i] = 0;
}

}  // namespace

// Rule for the rows' home.  Up to kResidentGains gains per block (two evaluations per thread) all of them are predicted
// at once, kept in shared memory and walked there; the whole table is written as well.  Beyond that prediction is what
// costs (910 us for 128 gains of a million jobs each), so rows start with four times the average number of
// cores handed out, at least 16, and only rows that need more are continued.  Large tables are predicted down to a bound from a
// sample instead (select_bounded).
constexpr int kKeepLast = 8192;
constexpr int kSmallGains = 6144, kSmallRows = 256;   // one block up to here (see select_small_kernel)

static size_t select_smem(bool curves, int rows, int stride) {
    return sizeof(double) * ((curves ? 7 * kThreads + kThreads / 2 : 0) + (size_t)rows * stride);
}

int select_setup(int* blocks_per_sm) {
    int per_sm = 1;
    const size_t most = select_smem(true, kKeepLast, 1), most_small = select_smem(true, kSmallGains + kSmallRows, 1);
    for (const void* k : {(const void*)select_small_kernel<true>, (const void*)select_small_kernel<false>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most_small) != cudaSuccess) return -1;
    for (const void* k : {(const void*)select_kernel<true, false, OneHandle>, (const void*)select_kernel<true, true, OneHandle>,
                          (const void*)select_kernel<false, false, OneHandle>, (const void*)select_kernel<true, false, ManyHandles>,
                          (const void*)select_kernel<true, true, ManyHandles>})
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most) != cudaSuccess) return -1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, select_kernel<true, true, ManyHandles>, kThreads, most) != cudaSuccess) return -1;
    *blocks_per_sm = per_sm < 1 ? 1 : per_sm;
    return 0;
}

// The part of the arguments that depends on the sizes, the same for all handles of a launch (J: their rows in all).
struct SelectPlan {
    int depth, W, rows, stride, keep_last, bounded;
    size_t smem;
};
static void set_rows(SelectPlan& p, int rows, int cap, bool curves) {
    p.rows = rows;
    p.keep_last = !p.bounded && p.stride == 0 && p.depth < cap && rows <= kKeepLast;
    p.smem = select_smem(curves, p.stride > 0 || p.keep_last ? rows : 0, p.stride > 0 ? p.stride : 1);
}
static SelectPlan plan_select(long long J, int cap, long long want, bool curves, int sm_count, int blocks_per_sm) {
    SelectPlan p;
    const long long gains = J * cap;
    p.depth = select_depth(J, cap, want, sm_count);
    p.bounded = curves && select_bounded(J, cap, want, sm_count, sm_count * blocks_per_sm);
    p.W = 1;
    long long grid;
    if (gains <= (long long)kResidentGains * sm_count) {
        while (p.W < 32 && p.W < cap) p.W <<= 1;
        grid = std::min<long long>(sm_count, std::max<long long>(1, (gains + kThreads - 1) / kThreads));
        p.stride = cap | 1;   // odd: threads walking neighbouring rows meet different banks
    } else {
        while (p.W < 16 && p.W < cap) p.W <<= 1;
        grid = (long long)sm_count * blocks_per_sm;
        p.stride = 0;
    }
    set_rows(p, (int)((J + grid - 1) / grid), cap, curves);
    return p;
}
static void apply_plan(SelectArgs& a, const SelectPlan& p) {
    a.depth = p.depth;
    a.W = p.W;
    a.rows = p.rows;
    a.stride = p.stride;
    a.keep_last = p.keep_last;
}

static bool one_block(long long J, int cap) { return J <= kSmallRows && J * cap <= kSmallGains; }

static cudaError_t launch_one(OneHandle& one, bool curves, int sm_count, int blocks_per_sm, cudaStream_t st) {
    SelectArgs& a = one.a;
    const SelectPlan p = plan_select(a.J, a.cap, a.want, curves, sm_count, blocks_per_sm);
    apply_plan(a, p);
    if (one_block(a.J, a.cap)) {
        const size_t smem = select_smem(curves, a.J, p.stride);
        return launch_behind(curves ? select_small_kernel<true> : select_small_kernel<false>, 1, kThreads, smem, st, one);
    }
    return launch_behind<true>(p.bounded ? select_kernel<true, true, OneHandle> : curves ? select_kernel<true, false, OneHandle> : select_kernel<false, false, OneHandle>, (a.J + p.rows - 1) / p.rows,
                               kThreads, p.smem, st, one);
}

static SelectArgs handle_args(slaq_handle* h, double epoch_seconds, long long want, int first_unit, int32_t* d_out_alloc, uint32_t seq) {
    SelectArgs a;
    a.job = h->job;
    a.fit = h->fit;
    a.count = h->job.count;
    a.gain = h->gain;
    a.J = h->max_jobs;
    a.cap = h->max_cores;
    a.first_unit = first_unit;
    a.T = epoch_seconds;
    a.want = want;
    a.gl = h->scratch.select;
    a.sel = h->scratch.sel;
    a.counters = h->scratch.counters;
    a.gt = h->scratch.gt;
    a.eq = h->scratch.eq;
    a.list = h->scratch.order;   // the fits are done with it
    a.alloc = h->alloc;
    a.last_alloc = h->job.last_alloc;
    a.out_alloc = d_out_alloc;
    a.reduction = h->reduction;
    a.err_word = h->err_word;
    a.basis = h->basis;
    a.zero = h->scratch.zero;
    a.zero_words = (int)(h->scratch.zero_bytes / sizeof(u64));
    a.published = h->scratch.published;
    a.mail = seq ? h->mailbox : nullptr;
    a.mail_alloc = seq && h->max_jobs <= h->mailbox_jobs ? h->mail_alloc() : nullptr;
    a.seq = seq;
    a.stamps = h->scratch.stamps;
    return a;
}

int launch_select(slaq_handle* h, double epoch_seconds, long long want, int first_unit, bool from_curves, int32_t* d_out_alloc,
                  uint32_t seq) {
    OneHandle one{handle_args(h, epoch_seconds, want, first_unit, d_out_alloc, seq)};
    const cudaError_t e = launch_one(one, from_curves, h->sm_count, h->select_blocks_per_sm, h->stream);
    if (e != cudaSuccess) {
        h->err = std::string("selection launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

int launch_select_group(slaq_handle* const* hs, int n, double epoch_seconds, long long want, int first_unit, uint32_t seq,
                        bool* whole_table) {
    slaq_handle* const h = hs[0];
    ManyHandles many;
    long long J = 0;
    for (int s = 0; s < n; ++s) J += hs[s]->max_jobs;
    SelectPlan p = plan_select(J, h->max_cores, want, true, h->sm_count, h->select_blocks_per_sm);
    // a handle's last block may be partly empty: a few more rows per block until all blocks are resident at once
    int blocks;
    for (int rows = p.rows;; ++rows) {
        blocks = 0;
        for (int s = 0; s < n; ++s) blocks += (hs[s]->max_jobs + rows - 1) / rows;
        set_rows(p, rows, h->max_cores, true);
        if (blocks <= h->sm_count * h->select_blocks_per_sm) break;
    }
    *whole_table = p.depth == h->max_cores;
    many.n = n;
    many.first_block[0] = 0;
    for (int s = 0; s < kMaxShards; ++s) {
        if (s < n) {
            SelectArgs& a = many.a[s];
            a = handle_args(hs[s], epoch_seconds, want, first_unit, nullptr, seq);
            a.gl = h->scratch.select;
            a.mail = h->mailbox;
            apply_plan(a, p);
        }
        many.first_block[s + 1] = many.first_block[s] + (s < n ? (hs[s]->max_jobs + p.rows - 1) / p.rows : 0);
    }
    const cudaError_t e = launch_behind<true>(p.bounded ? select_kernel<true, true, ManyHandles> : select_kernel<true, false, ManyHandles>, blocks, kThreads, p.smem, h->stream, many);
    if (e != cudaSuccess) {
        h->err = std::string("selection launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

bool select_writes_whole_table(const slaq_handle* h, long long want) {
    return select_depth(h->max_jobs, h->max_cores, want, h->sm_count) == h->max_cores;
}

// ---------------------------------------------------------------------------------
// Allocation without any device allocation: the same kernel, its scratch in a static device array that ships with the
// library image.
// ---------------------------------------------------------------------------------
namespace {

constexpr int kStaticMaxJobs = 32768;

struct StaticScratch {
    SelectGlobal gl;                 // its leading part is cleared every call
    SelectState sel;                 // rewritten every call
    long long counters[16];
    int32_t gt[kStaticMaxJobs], eq[kStaticMaxJobs];   // written before they are read
};

static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

struct StaticDevice {
    StaticScratch* scratch;
    int sm_count, blocks_per_sm;
};

// Device address of g_static_scratch on the current device and its launch limits, looked up once per device.
// In host code the array's name only stands for the symbol; kernels need this address.
int static_scratch_for_current_device(StaticDevice* out) {
    constexpr int kMaxDevices = 64;
    static StaticDevice cache[kMaxDevices] = {};
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return SLAQ_E_CUDA;
    StaticScratch* p = __atomic_load_n(&cache[dev].scratch, __ATOMIC_ACQUIRE);
    if (!p) {
        void* addr = nullptr;
        int sm = 0, per_sm = 1;
        if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || !addr) return SLAQ_E_CUDA;
        if (cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return SLAQ_E_CUDA;
        if (select_setup(&per_sm)) return SLAQ_E_CUDA;
        p = static_cast<StaticScratch*>(addr);
        __atomic_store_n(&cache[dev].sm_count, sm, __ATOMIC_RELAXED);
        __atomic_store_n(&cache[dev].blocks_per_sm, per_sm, __ATOMIC_RELAXED);
        __atomic_store_n(&cache[dev].scratch, p, __ATOMIC_RELEASE);   // every thread finds the same values
    }
    out->scratch = p;
    out->sm_count = __atomic_load_n(&cache[dev].sm_count, __ATOMIC_RELAXED);
    out->blocks_per_sm = __atomic_load_n(&cache[dev].blocks_per_sm, __ATOMIC_RELAXED);
    return SLAQ_OK;
}

}  // namespace

}  // namespace slaq

extern "C" int slaq_allocate_static(const double* d_gain, int32_t n_jobs, int32_t max_cores_per_job,
                                    int64_t total_cores, int32_t* d_out_alloc, double* d_out_reduction,
                                    void* cuda_stream) {
    using namespace slaq;
    if (!d_gain || !d_out_alloc || !d_out_reduction || n_jobs < 1 || max_cores_per_job < 1 || total_cores < 0)
        return SLAQ_E_ARG;
    if (n_jobs > kStaticMaxJobs || max_cores_per_job > kMaxCoresLimit) return SLAQ_E_RANGE;
    StaticDevice dev;
    const int rc = static_scratch_for_current_device(&dev);
    if (rc) return rc;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int J = n_jobs, cap = max_cores_per_job;
    const int floor_units = total_cores >= J ? 1 : 0;
    const long long usable = total_cores < (long long)J * cap ? total_cores : (long long)J * cap;
    // the array keeps the previous call's contents: clear what the kernel accumulates into
    if (!one_block(J, cap) && cudaMemsetAsync(&dev.scratch->gl, 0, SelectGlobal::kZeroBytes, st) != cudaSuccess) return SLAQ_E_CUDA;
    OneHandle one = {};
    SelectArgs& a = one.a;
    a.gain = const_cast<double*>(d_gain);   // only read: no gains are predicted here
    a.J = J;
    a.cap = cap;
    a.first_unit = floor_units + 1;
    a.want = usable - (long long)J * floor_units;
    a.gl = &dev.scratch->gl;
    a.sel = &dev.scratch->sel;
    a.counters = dev.scratch->counters;
    a.gt = dev.scratch->gt;
    a.eq = dev.scratch->eq;
    a.alloc = d_out_alloc;
    a.reduction = d_out_reduction;
    if (launch_one(one, false, dev.sm_count, dev.blocks_per_sm, st) != cudaSuccess) return SLAQ_E_CUDA;
    if (total_cores < J) return SLAQ_W_OVERSUBSCRIBED;
    if (total_cores > (long long)J * cap) return SLAQ_W_UNDERFILLED;
    return SLAQ_OK;
}
