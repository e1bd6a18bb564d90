// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "slaq.h"
#include "slaq_bounds.cuh"
#include "slaq_fit_plan.cuh"

namespace slaq {

constexpr int kMaxHistLimit = 6000;   // one warp stages a whole window in shared memory
constexpr int kMaxCoresLimit = 1024;
constexpr int kRadixBits = 11;
constexpr int kRadixBins = 1 << kRadixBits;
constexpr int kRadixPasses = 6;       // 11 + 11 + 11 + 11 + 11 + 9 bits, most significant first
constexpr int kFitQueueBase = 8;      // ticket[kFitQueueBase + c]: work queue head of class c
constexpr int kTickets = 16;

// Device-side state of one job, structure of arrays (index = job id).
struct JobArrays {
    double** row;        // start of the job's window storage (ring of `cap` slots)
    int32_t* cap;        // slots in the ring
    int32_t* head;       // slot the next loss goes to
    int32_t* count;      // stored losses, 0 = inactive
    int64_t* k_last;     // iteration index of the newest loss
    double* m_seen;      // largest one-step reduction seen so far (-inf: none)
    double* tm;          // [8][max_jobs]: count, sum u, sum u^2, sum t, sum u t, sum t n, min u, max u (u = 1/cores)
    double* s_set;       // fixed time law (NaN: use the estimate)
    double* w_set;
    int32_t* last_alloc; // core count of the last epoch (1 before any)
    double* target;      // hint of the loss the job will end at (NaN: none)
    // extents, read by the bounds build only
    int32_t max_jobs;
    const double* ring_lo;     // the ring pool [ring_lo, ring_hi)
    const double* ring_hi;
    const double* packed_lo;   // the packed pool (both null while there is none)
    const double* packed_hi;
    int32_t* err_word;
};

// What the fit leaves for the later stages, one entry per job.
struct FitArrays {
    int32_t* status;     // SLAQ_JOB_*
    int8_t* family;      // 0, 1 or -1
    double* params;      // [max_jobs][4]; linear-extrapolation kinds keep (rho, r_cap) in slots 0, 1
    double* residual;    // [max_jobs][2]
    int32_t* sweeps;     // [max_jobs][2]
    double* largest;     // M
    double* span;        // max(H-1, 1)
    // Both families' end points of the last epoch, in that epoch's window coordinates
    // (span, largest and k_fit say which), and the copy the next fit may start from.  A
    // job's copy is refreshed when its history changes, so an epoch repeated without new
    // losses starts from the same point and gives the same result.
    double* both;        // [max_jobs][8]: family I (a, b, c, d), family II (alpha, beta, c, unused)
    uint8_t* mask;       // bit 0 / 1: family I / II ended with a finite residual
    int64_t* k_fit;      // index of the newest iteration at that fit
    double* warm_p;      // [max_jobs][8]
    uint8_t* warm_mask;
    int64_t* warm_k;
    double* warm_span;
    double* warm_scale;
};

// What the last epoch's gain rows follow from.  An epoch writes rows of a large table only as far as its selection needs them;
// asked for later they must still be that epoch's, whatever has happened to the time laws, the hints or the fits since.  So
// such an epoch keeps its curves: 49 bytes per job, against 8 max_cores_per_job for the rows themselves.
struct GainNote {
    int32_t partial;     // the rows are written only in part, and the curves below are those they follow from
    int32_t cap;         // entries of a row
    double T;
};
struct GainBasis {
    double* v;           // [6][max_jobs]: the curve's three parameters, 1 / span, s, w
    int8_t* kind;        // [max_jobs]
    GainNote* note;
};

// Running state of the radix select.
struct SelectState {
    unsigned long long prefix;       // bits of the threshold key found so far
    long long want;                  // units still to take inside the current candidate set
    int done;                        // nothing is wanted: the threshold lies above every gain
};

constexpr int kSelectFineBins = 2048;
constexpr int kSelectCandidates = 2048;
constexpr int kSelectMaxGrid = 4096;

// Global memory of the selection launch.  The leading part is cleared before every launch.
struct SelectGlobal {
    unsigned long long fine[kSelectFineBins];             // first histogram: 64 bins per power of two
    unsigned int barrier, ticket, n_cand, sampled;        // blocks that arrived; blocks that finished; listed candidates; rows in the sample
    static constexpr size_t kZeroBytes = sizeof(unsigned long long) * kSelectFineBins + 16;
    // cleared by the kernel itself: later histograms, apart from the first one, which slower blocks may still be reading when
    // the first of these counts arrive; the histograms of the narrowing steps
    unsigned long long fine_more[kSelectFineBins], fine_rest[kSelectFineBins];
    unsigned long long narrow[kRadixPasses][kRadixBins];
    unsigned long long cand_key[kSelectCandidates];       // the candidates the last block ranks ..
    unsigned long long cand_pos[kSelectCandidates];       // .. and their (candidates of the row, job, n)
    long long block_eq[kSelectMaxGrid];                   // per block: candidates that equal the threshold
};

// Page-locked host memory of a handle that kernels write and read directly: a call is over when `done` holds its number.
struct Mailbox {
    volatile uint32_t done;
    volatile int32_t err;            // the device error word when the call finished; a bulk load: a loss is not finite
    volatile int64_t points;         // state export: stored losses in all, and the longest window
    volatile int32_t longest;
    uint32_t pad[11];
};
constexpr int32_t kMailboxJobs = 32768;   // most entries per call that pass through the mailbox's arrays

// Scratch of one epoch.  [zero, zero + zero_bytes) is cleared at the start of every epoch; the sharded steps
// clear their histograms `hist` as well.
struct Scratch {
    unsigned long long* hist;        // [kRadixPasses][kRadixBins], sharded steps
    void* zero;
    SelectGlobal* select;            // its leading part is the end of the cleared region
    unsigned int* ticket;            // [kTickets]: work queue of the fit
    SelectState* sel;
    long long* counters;             // [16] statistics accumulated by kernels during an epoch
    long long* published;            // [16] those of the last finished epoch
    long long* stamps;               // [4] behind `published`: device clock (ns) when its first kernel, the gain kernel and the selection started, and at its end
    unsigned int* append_ticket;     // blocks of a reporting kernel that are done
    int32_t* load_flag;              // a bulk load brought a loss that is not finite
    size_t zero_bytes;
    int32_t* gt;                     // per job: during the passes the start of its candidate segment, then gains above the threshold
    int32_t* eq;                     // per job: during the passes the end of its segment, then gains equal to the threshold
    long long* block_eq;             // per block of the count kernel: sum of eq
    int32_t* bucket;                 // [max_hist + 1] jobs per window length (inside the cleared region)
    int32_t* order;                  // job ids, longest window first (fit kernel work list)
    int32_t* start;                  // [max_hist + 1] start[h] = jobs with a window longer than h
    int32_t* cursor;                 // [max_hist + 1] scatter positions of the counting sort
};

struct Staging {
    int32_t* ids;
    double* losses;
    double* times;
    int32_t* cores;
    int64_t* offsets;
    int64_t* k_last;
    double* m_seen;
};

}  // namespace slaq

struct slaq_handle {
    int device = 0;
    int32_t max_jobs = 0, max_hist = 0, cap_alloc = 0;   // cap_alloc: gain columns the buffers were sized for
    int32_t max_cores = 64;
    double gamma = 0.9;
    int32_t lm_trials = 20, min_fit_points = 4;
    size_t fit_slice_bytes = slaq::kDefaultFitSlice;   // shared memory one warp of the fit kernel may use (parked sums, rows of 32 points, a spare row); the default: by size
    bool warm_start = false;              // fits start from the last epoch's parameters where there are some
    int selection = 0;                    // SLAQ_P_SELECTION: kept for callers that ask, read by nothing else
    bool gain_partial = false;            // h->gain holds the last epoch's rows only in part (see GainBasis)
    bool epoch_captured = false;          // an epoch of the handle is part of a graph of the caller: only the device knows which was last
    std::vector<uint8_t> hinted;          // host mirror: job has a target-loss hint
    int32_t n_hinted = 0;
    bool gain_envelope = false;           // gain rows are slopes of the concave envelope of R(n), not a running minimum
    int64_t fit_cluster_jobs = 0;         // active jobs the lanes per job are chosen for (0: this handle's own)
    cudaStream_t stream = nullptr;
    bool owns_ws = false;
    void* ws = nullptr;
    size_t ws_bytes = 0;
    double* ring_pool = nullptr;      // [max_jobs][max_hist]
    double* packed_pool = nullptr;    // separate allocation made by slaq_load_histories_packed
    size_t packed_len = 0;
    void* call_buf = nullptr;         // scratch of calls that move caller data of any size (grown on demand, kept)
    size_t call_buf_bytes = 0;
    double* wtab = nullptr;           // gamma^m, m = 0..max_hist-1, then the sums over m < H of gamma^m m^p: [5][max_hist + 1], then (16-byte aligned) the logarithm's table
    double wtab_gamma = -1.0;
    slaq::JobArrays job;
    slaq::FitArrays fit;
    slaq::GainBasis basis;
    slaq::Scratch scratch;
    slaq::Staging stage;
    double* gain = nullptr;           // [max_jobs][max_cores]
    int32_t* alloc = nullptr;
    double* reduction = nullptr;
    int32_t* err_word = nullptr;      // device error flags set by kernels
    bool pipe_user = false;           // counted among the users of the bulk copies' buffers
    void* mailbox_mem = nullptr;      // page-locked: Mailbox, then ids, losses, times, cores in and the allocation out
    slaq::Mailbox* mailbox = nullptr;
    int32_t mailbox_jobs = 0;         // entries of each of those arrays
    int32_t* mail_ids() const { return reinterpret_cast<int32_t*>(mailbox + 1); }
    int32_t* mail_cores() const { return mail_ids() + mailbox_jobs; }
    int32_t* mail_alloc() const { return mail_cores() + mailbox_jobs; }
    double* mail_losses() const { return reinterpret_cast<double*>(mail_alloc() + mailbox_jobs + (mailbox_jobs & 1)); }
    double* mail_times() const { return mail_losses() + mailbox_jobs; }
    uint32_t call_seq = 0;            // number of the last call that reports to the mailbox
    uint32_t mail_seq = 0;            // number of the append that reads its entries from the mailbox's arrays
    bool mail_in_use = false;         // and whether it may still be reading them
    bool scratch_clean = false;       // the last epoch left its scratch cleared for the next one
    cudaEvent_t ev[4] = {};               // stage boundaries of the sharded steps and of replayed graphs
    cudaEvent_t order_ev[2] = {};         // fork and join of fits that run beside one another
    cudaEvent_t order_event(int i) {
        if (!order_ev[i] && cudaEventCreateWithFlags(&order_ev[i], cudaEventDisableTiming) != cudaSuccess) order_ev[i] = nullptr;
        return order_ev[i];
    }
    bool have_epoch = false;
    int32_t last_launches = 0;            // kernels the last call launched
    int select_blocks_per_sm = 1;         // resident blocks of the selection kernel
    const void* fit_ready = nullptr;      // the fit kernel whose shared memory was allowed last
    int sm_count = 148;
    std::vector<uint8_t> active;      // host mirror: job has at least one loss
    std::vector<uint32_t> stamp;      // host: duplicate detection
    std::vector<uint8_t> in_packed;   // host: job's row lives in the packed pool
    uint32_t stamp_epoch = 0;
    int32_t n_active = 0;
    int shard_first_unit = 2;         // set by slaq_shard_predict for the steps that follow
    // The epoch as a CUDA graph: what the captured launches depended on, the instantiated graph,
    // and the stream the capture runs on (the caller's stream may be the legacy default stream,
    // which cannot capture).
    int epoch_graph = -1;             // 1: replay the launches as a graph; 0, -1: plain launches
    std::vector<long long> graph_key, seen_key;
    cudaGraphExec_t graph_exec = nullptr;
    cudaStream_t capture_stream = nullptr;
    cudaStream_t side_stream = nullptr;   // the fit of a handle that is scheduled together with others
    int32_t graph_launches = 0;
    bool last_epoch_was_graph = false;
    bool last_gain_launch = false;        // it had a gain kernel of its own
    bool last_fit_launch = false;         // and a fit
    std::string err;
};

namespace slaq {

// ---- launches of an epoch ----
//
// An epoch is two to five launches in a row, and at small sizes the gaps between them count: 8 us of a pass of 70 to 170 us were
// four timing events between the launches, so the kernels note the device clock themselves, and a kernel that follows another
// is launched while that one still runs (its blocks wait at after_previous() before they touch what it leaves).
__device__ __forceinline__ void note_time(long long* stamp) {
    if (stamp && blockIdx.x == 0 && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
        *stamp = (long long)t;
    }
}
// Everything the kernels before this one wrote is visible behind this line; the kernel after this one may be launched.
__device__ __forceinline__ void after_previous() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <bool kCooperative = false, class... Params, class... Args>
cudaError_t launch_behind(void (*kernel)(Params...), int blocks, int threads, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = kCooperative ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// kernel launchers: each returns the number of kernels it launched, or -1 after setting h->err
int fit_prepare(slaq_handle* h);   // loads what a fit of all the handle's ids launches; 0 or -1
// on `st`, with at most max_blocks blocks
int launch_fit(slaq_handle* h, cudaStream_t st, int max_blocks);
int fit_least_lanes(const slaq_handle* h);
// histogram: the keys go into scratch.hist's first pass as well
int launch_gain(slaq_handle* h, double epoch_seconds, int first_unit, bool histogram);
// the rest of the last epoch's rows, from the curves it kept; does nothing if the rows are whole
int launch_complete_gains(slaq_handle* h);
// seq != 0: the kernel reports to the handle's mailbox under that number, and writes the allocation there too if it fits
int launch_select(slaq_handle* h, double epoch_seconds, long long want, int first_unit, bool from_curves, int32_t* d_out_alloc,
                  uint32_t seq);
// one cluster whose jobs are held by n handles of this GPU (n <= kMaxGroup), on the first one's stream; reports to its mailbox
constexpr int kMaxGroup = 8;
int launch_select_group(slaq_handle* const* hs, int n, double epoch_seconds, long long want, int first_unit, uint32_t seq,
                        bool* whole_table);
bool select_writes_whole_table(const slaq_handle* h, long long want);
int select_setup(int* blocks_per_sm);   // before a handle's first selection launch; 0 or -1
int launch_normalise_export(slaq_handle* h, int32_t n, const int64_t* d_offsets, double* d_changes,
                            double* d_levels, double* d_largest);
int launch_time_model(slaq_handle* h, double* d_s, double* d_w);
int launch_shard_pick(slaq_handle* h, int pass, long long want);
int launch_shard_pass(slaq_handle* h, int pass, int first_unit);
int launch_shard_count(slaq_handle* h, int first_unit, const long long** d_total);
int launch_shard_finalise(slaq_handle* h, int first_unit, long long ties_before, const long long* d_ties_before,
                          int32_t* d_out_alloc);

}  // namespace slaq
