// Marginal gains: expand every job's fitted curve into the predicted loss reduction of its
// n-th core, n = 1..max_cores_per_job (the objective Loss_j(a_j, t) - Loss_j(a_j, t+T) of
// "Scheduling Based on Quality Improvements", differenced in a_j).
//
// An iteration on n cores takes t(n) = s + w/n seconds, so an epoch of T seconds runs
// m(n) = T n / (s n + w) iterations; in window coordinates that is X_n = m(n) / span ahead
// of the newest point, and R(n) = f(0) - f(X_n).  g(n) = R(n) - R(n-1) is evaluated without
// cancellation (divisions by Newton reciprocals: a gain is good to a few ulp), clamped to +0
// where it is not a positive finite number, and made non-increasing in n by a running minimum.  A job has W lanes, the
// power of two that covers its row, 32 at most; the row is written once, coalesced.  The sharded steps take the first
// histogram of the threshold selection from here as well.
#include <math_constants.h>

#include <algorithm>

#include "slaq_internal.cuh"
#include "slaq_gain_curve.cuh"

namespace slaq {

namespace {

using namespace gaincurve;

constexpr int kThreads = 256;

// Slopes of the upper concave envelope of the points (n, R(n)), n = 0..cap, written over the row
// (row[n-1] holds the clamped difference R(n) - R(n-1) on entry).  One thread walks the row: a stack
// of envelope vertices, a point leaving it when it lies on or below the chord from the vertex
// before it to the new point.  Rows that need this are rare (the fit is not convex ahead), and one thread's chain of
// loads is what they cost, so the row lies in shared memory.
__device__ void envelope_of_row(double* row, int cap, unsigned short* stack) {
    double run = 0.0;
    for (int n = 1; n <= cap; ++n) {   // differences -> R(n) in place
        run += row[n - 1];
        row[n - 1] = run;
    }
    auto R = [&](int n) { return n == 0 ? 0.0 : row[n - 1]; };
    int top = 0;
    for (int n = 0; n <= cap; ++n) {
        while (top >= 2) {
            const int a = stack[top - 2], b = stack[top - 1];
            if ((R(b) - R(a)) * (double)(n - b) <= (R(n) - R(b)) * (double)(b - a)) --top;
            else break;
        }
        stack[top++] = (unsigned short)n;
    }
    // slopes, written from the right so that R(a) of each segment is still in place when it is read
    for (int v = top - 1; v >= 1; --v) {
        const int a = stack[v - 1], b = stack[v];
        const double slope = (R(b) - R(a)) / (double)(b - a);
        for (int n = b; n > a; --n) row[n - 1] = slope;
    }
}

// A lane's key into the block's histogram; lanes with equal digits add once.
__device__ __forceinline__ void count_key(unsigned int* hist, double g, bool counted, int32_t* err_word) {
    const unsigned digit = (unsigned)((unsigned long long)__double_as_longlong(g) >> (64 - kRadixBits));
    const unsigned live = __ballot_sync(kFull, counted);
    if (counted) {
        const unsigned peers = __match_any_sync(live, digit);
        if ((int)(__ffs(peers) - 1) == (int)(threadIdx.x & 31) && index_ok(digit, kRadixBins, kErrBin, err_word))
            atomicAdd(&hist[digit], (unsigned)__popc(peers));
    }
}

// kKept: the rows of the last epoch from the curves it kept (see GainBasis), where it has left them unfinished.
// kOptions: the instantiation that knows the two options of the prediction (the plain one carries none of
// their code).  envelope: rows become the slopes of the concave envelope of R(n) instead of a
// running minimum; target-loss hints are read per job.  hist0: null where nobody reads the histogram.
//
// What bounds it is latency, of one row's steps (load the curve, predict, envelope, cap) where jobs are few, of all rows'
// where they are many.  With a warp per job whatever its row's length, and the envelope walked in global memory, 4,000
// rows of 64 took 35 us (now 31) and 542,000 rows of 5 took 370 (now 130).
template <bool kOptions, bool kKept>
__global__ void __launch_bounds__(kThreads, 5)
gain_kernel(JobArrays job, FitArrays fit, GainBasis basis, int max_jobs, int cap, int W, double T, int first_unit, double* __restrict__ gain,
            long long* stamp, unsigned long long* __restrict__ hist0, bool envelope) {
    extern __shared__ double dyn[];      // kOptions: [groups][cap] rows, then [groups][cap + 1] vertices
    __shared__ unsigned int sh_hist[kRadixBins];
    after_previous();
    if (kKept) {
        const GainNote note = *basis.note;
        if (!note.partial) return;
        cap = note.cap;
        T = note.T;
    } else {
        note_time(stamp);
        if (blockIdx.x == 0 && threadIdx.x == 0) *basis.note = GainNote{0, cap, T};
    }
    if (hist0) {
        for (int i = threadIdx.x; i < kRadixBins; i += kThreads) sh_hist[i] = 0;
        __syncthreads();
    }
    const int groups = kThreads / W, group = threadIdx.x / W, w = threadIdx.x & (W - 1);
    for (int base = blockIdx.x * groups; base < max_jobs; base += gridDim.x * groups) {   // uniform: the steps use warp shuffles
        const int j = base + group;
        const bool in = j < max_jobs;
        const bool active = in && job.count[j] > 0;
        bool no_time = false;
        Curve c = {};
        c.kind = 3;
        if (in) c = kKept ? kept_curve(basis, j, max_jobs, T) : load_curve<true>(job, fit, j, max_jobs, T, &no_time);
        if (no_time && w == 0) fit.status[j] = SLAQ_JOB_NO_TIME;
        double* const out = gain + (size_t)(in ? j : 0) * cap;
        double* const row = kOptions ? dyn + (size_t)group * cap : out;
        double carry = CUDART_INF;   // (smallest) gain before this chunk
        int rises = 0;
        for (int n0 = 0; n0 < cap; n0 += W) {
            const int n = n0 + w + 1;
            const bool has = in && n <= cap && index_ok((long long)j * cap + (n - 1), (long long)max_jobs * cap, kErrGain, job.err_word);
            double g = CUDART_INF;
            if (has) g = c.kind == 3 ? 0.0 : raw_gain(c, n);
            // inclusive running minimum over n; most chunks fall already (convex fits), which one look at the
            // left neighbour shows
            double left = __shfl_up_sync(kFull, g, 1, W);
            if (w == 0) left = carry;
            if (kOptions && envelope) {
                rises |= (has && g > left) ? 1 : 0;
            } else if (__any_sync(kFull, has && g > left)) {
                for (int o = 1; o < W; o <<= 1) {
                    const double up = __shfl_up_sync(kFull, g, o, W);
                    if (w >= o) g = fmin(g, up);
                }
                g = fmin(g, carry);
            }
            carry = __shfl_sync(kFull, g, W - 1, W);
            if (has) row[n - 1] = g;
            if (!kOptions && hist0) count_key(sh_hist, g, has && active && n >= first_unit, job.err_word);
        }
        if (!kOptions) continue;
        // A target-loss hint caps the predicted reduction at (newest loss - target) / M.
        double reduction_cap = CUDART_INF;
        if (c.kind != 3) {
            const double target = job.target[j];
            const double M = fit.largest[j];
            if (finite_d(target) && M > 0.0) {
                const int ring = job.cap[j];
                int at = job.head[j] - 1;
                at += at < 0 ? ring : 0;
                const double newest = index_ok(at, ring, kErrStorage, job.err_word) ? job.row[j][at] : 0.0;
                reduction_cap = __ddiv_rn(fmax(newest - target, 0.0), M);
            }
        }
        __syncwarp();
        if (envelope) {
            for (int o = W >> 1; o > 0; o >>= 1) rises |= __shfl_xor_sync(kFull, rises, o);
            if (rises && w == 0)
                envelope_of_row(row, cap, reinterpret_cast<unsigned short*>(dyn + (size_t)groups * cap) + (size_t)group * (cap + 1));
            __syncwarp();
        }
        const bool capped = __any_sync(kFull, reduction_cap < CUDART_INF);
        double before = 0.0;   // uncapped reduction of the cores before this chunk
        for (int n0 = 0; n0 < cap; n0 += W) {
            const int n = n0 + w + 1;
            const bool has = in && n <= cap;
            double g = has ? row[n - 1] : 0.0;
            if (capped) {
                double incl = g;
                for (int o = 1; o < W; o <<= 1) {
                    const double up = __shfl_up_sync(kFull, incl, o, W);
                    if (w >= o) incl += up;
                }
                const double left = reduction_cap - (before + (incl - g));
                before += __shfl_sync(kFull, incl, W - 1, W);
                if (reduction_cap < CUDART_INF) g = left > 0.0 ? fmin(g, left) : 0.0;
            }
            if (has) out[n - 1] = g;
            if (hist0) count_key(sh_hist, g, has && active && n >= first_unit, job.err_word);
        }
        __syncwarp();   // the row is read before the next job's is written
    }
    if (!hist0) return;
    __syncthreads();
    for (int i = threadIdx.x; i < kRadixBins; i += kThreads) {
        const unsigned v = sh_hist[i];
        if (v) atomicAdd(&hist0[i], (unsigned long long)v);
    }
}

__global__ void time_model_kernel(JobArrays job, int max_jobs, double* out_s, double* out_w) {
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= max_jobs) return;
    double s = CUDART_NAN, w = CUDART_NAN;
    (void)time_law(job, j, max_jobs, s, w);   // leaves NaN where the job has neither a fixed law nor samples
    out_s[j] = s;
    out_w[j] = w;
}

}  // namespace

int launch_gain(slaq_handle* h, double epoch_seconds, int first_unit, bool histogram) {
    const int J = h->max_jobs, cap = h->max_cores;
    int W = 1;
    while (W < 32 && W < cap) W <<= 1;
    const int groups = kThreads / W;
    const bool options = h->gain_envelope || h->n_hinted > 0;
    const size_t smem = options ? (size_t)groups * (sizeof(double) * cap + sizeof(unsigned short) * (cap + 1)) : 0;
    const auto kernel = options ? gain_kernel<true, false> : gain_kernel<false, false>;
    cudaError_t e = cudaSuccess;
    int per_sm = 5;
    if (smem > 32 * 1024) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        per_sm = 2;
    }
    const int blocks = std::min(h->sm_count * per_sm, (J + groups - 1) / groups);
    if (e == cudaSuccess)
        e = launch_behind(kernel, blocks, kThreads, smem, h->stream, h->job, h->fit, h->basis, J, cap, W, epoch_seconds, first_unit,
                          h->gain, h->scratch.stamps + 1, histogram ? h->scratch.hist : nullptr, h->gain_envelope);
    if (e != cudaSuccess) {
        h->err = std::string("gain kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

int launch_complete_gains(slaq_handle* h) {
    const int J = h->max_jobs, cap = h->max_cores;   // the epoch's own cap is in its note; this one decides the lanes per row
    int W = 1;
    while (W < 32 && W < cap) W <<= 1;
    const int groups = kThreads / W, blocks = std::min(h->sm_count * 5, (J + groups - 1) / groups);
    gain_kernel<false, true><<<blocks, kThreads, 0, h->stream>>>(h->job, h->fit, h->basis, J, cap, W, 0.0, 2, h->gain, nullptr, nullptr, false);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        h->err = std::string("gain kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

int launch_time_model(slaq_handle* h, double* d_s, double* d_w) {
    const int threads = 256, blocks = (h->max_jobs + threads - 1) / threads;
    time_model_kernel<<<blocks, threads, 0, h->stream>>>(h->job, h->max_jobs, d_s, d_w);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        h->err = std::string("time model kernel launch: ") + cudaGetErrorString(e);
        return -1;
    }
    return 1;
}

}  // namespace slaq
