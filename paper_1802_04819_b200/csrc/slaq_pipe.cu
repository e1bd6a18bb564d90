// Bulk copies between ordinary (pageable) host memory and the device.
//
// The driver moves pageable memory through its own staging buffer with one thread, at 6 to 10 GB/s, several times below
// what the link does.  Here up to kPipeThreads threads each take every n-th chunk, copy it into (or out of) one of their
// two page-locked buffers and queue the transfer of that buffer, so that copies of one chunk run beside transfers of
// others.  16 MB to the device: 1,530 us by cudaMemcpyAsync, 530 us with 4 threads and chunks of 1 MB (640 us with 512 KB,
// 850 us with 256 KB: a chunk's event and queueing cost more than its copy then), 313 us from page-locked memory, which
// is handed to the copy engine as it is.  Below kPipeFrom bytes starting threads costs more than it gives and the
// driver's path is taken.
//
// Page-locking costs milliseconds, which a process that loads once should not pay.  So the buffers are made once
// kPipeEarned bytes have gone (or are about to go) the slow way, and a result block once kResultEarned requests of its
// size have been answered with ordinary memory: about when they would have paid for themselves.
#include "slaq_pipe.cuh"

#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include "slaq_internal.cuh"

namespace slaq {

namespace {

constexpr int kPipeThreads = 4, kPipeBuffers = 2;
constexpr size_t kPipeChunk = 1024 * 1024, kPipeLeastChunk = 256 * 1024;
constexpr size_t kPipeEarned = 64 << 20;
constexpr int kResultEarned = 8;
constexpr size_t kResultBytes = 64 << 20, kResultLeast = 64 << 10;
constexpr size_t kPipeFrom = 256 * 1024;

struct Pool {
    std::mutex lock;         // one bulk copy of the process at a time uses the buffers
    std::mutex count_lock;
    int handles = 0;
    char* memory = nullptr;
    size_t earned = 0;       // bytes that went the driver's way (guarded by lock)
    std::map<size_t, int> asked;   // requests for result blocks by size, answered with ordinary memory
    // result blocks by address (guarded by count_lock)
    struct Block {
        size_t bytes;
        bool taken;
    };
    std::map<const char*, Block> blocks;
    size_t block_bytes = 0;
    // device memory that handles left behind, for the next ones' call buffers (guarded by count_lock)
    struct Spare {
        int device;
        void* memory;
        size_t bytes;
    };
    std::vector<Spare> spares;
};

Pool& pool() {
    static Pool p;
    return p;
}

bool page_locked(const void* p) {
    cudaPointerAttributes attr;
    if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return attr.type == cudaMemoryTypeHost;
}

int failed(slaq_handle* h, cudaError_t e) {
    h->err = std::string("bulk copy: ") + cudaGetErrorString(e);
    return SLAQ_E_CUDA;
}

// Copies chunk after chunk of one direction; what `thread` of `threads` does.
void work(slaq_handle* h, const std::vector<Segment>& chunks, bool down, int thread, int threads, std::atomic<int>& error) {
    cudaError_t e = cudaSetDevice(h->device);   // a new thread starts on device 0
    cudaEvent_t done[kPipeBuffers] = {};
    for (int b = 0; b < kPipeBuffers && e == cudaSuccess; ++b) e = cudaEventCreateWithFlags(&done[b], cudaEventDisableTiming);
    char* const base = pool().memory + (size_t)thread * kPipeBuffers * kPipeChunk;
    const Segment* flying[kPipeBuffers] = {};   // chunk whose transfer was last queued on each buffer
    int b = 0;
    auto land = [&](int k) {                    // wait for a buffer's transfer; downwards, empty it
        if (!flying[k]) return;
        e = cudaEventSynchronize(done[k]);
        if (e == cudaSuccess && down) std::memcpy(flying[k]->dst, base + k * kPipeChunk, flying[k]->bytes);
        flying[k] = nullptr;
    };
    for (size_t c = thread; c < chunks.size() && e == cudaSuccess && !error.load(); c += threads, b = (b + 1) % kPipeBuffers) {
        char* const buffer = base + b * kPipeChunk;
        land(b);
        if (e != cudaSuccess) break;
        if (!down) std::memcpy(buffer, chunks[c].src, chunks[c].bytes);
        e = down ? cudaMemcpyAsync(buffer, chunks[c].src, chunks[c].bytes, cudaMemcpyDeviceToHost, h->stream)
                 : cudaMemcpyAsync(chunks[c].dst, buffer, chunks[c].bytes, cudaMemcpyHostToDevice, h->stream);
        if (e == cudaSuccess) e = cudaEventRecord(done[b], h->stream);
        flying[b] = &chunks[c];
    }
    for (int k = 0; k < kPipeBuffers && e == cudaSuccess; ++k, b = (b + 1) % kPipeBuffers) land(b);   // the buffers are free again
    for (cudaEvent_t d : done)
        if (d) cudaEventDestroy(d);
    if (e != cudaSuccess) error.store((int)e);
}

int copy(slaq_handle* h, Segments segments, bool down) {
    std::vector<Segment> pageable;
    size_t total = 0;
    for (const Segment& s : segments) {
        const void* const host = down ? s.dst : s.src;
        if (s.bytes == 0 || !host) continue;
        if (s.bytes >= kPipeFrom && page_locked(host)) {
            const cudaError_t e = cudaMemcpyAsync(s.dst, s.src, s.bytes, down ? cudaMemcpyDeviceToHost : cudaMemcpyHostToDevice, h->stream);
            if (e != cudaSuccess) return failed(h, e);
            continue;
        }
        total += s.bytes;
        pageable.push_back(s);
    }
    Pool& p = pool();
    std::unique_lock<std::mutex> hold(p.lock, std::defer_lock);
    if (total >= kPipeFrom) {
        hold.lock();
        p.earned += p.memory ? 0 : total;
        if (!p.memory && p.earned >= kPipeEarned) {
            p.earned = 0;
            p.memory = static_cast<char*>(page_locked_alloc(kPipeThreads * kPipeBuffers * kPipeChunk));
        }
    }
    if (total < kPipeFrom || !p.memory) {
        for (const Segment& s : pageable) {
            const cudaError_t e = cudaMemcpyAsync(s.dst, s.src, s.bytes, down ? cudaMemcpyDeviceToHost : cudaMemcpyHostToDevice, h->stream);
            if (e != cudaSuccess) return failed(h, e);
        }
    } else {
        const size_t share = (total / (2 * kPipeThreads) + 4095) / 4096 * 4096;   // two chunks per thread, within limits
        const size_t chunk = std::min(kPipeChunk, std::max(kPipeLeastChunk, share));
        std::vector<Segment> chunks;
        for (const Segment& s : pageable)
            for (size_t at = 0; at < s.bytes; at += chunk)
                chunks.push_back({static_cast<char*>(s.dst) + at, static_cast<const char*>(s.src) + at, std::min(chunk, s.bytes - at)});
        const int cores = std::max(1, (int)std::thread::hardware_concurrency());
        const int threads = (int)std::min<size_t>({(size_t)kPipeThreads, (size_t)cores, (total + kPipeFrom - 1) / kPipeFrom, chunks.size()});
        std::atomic<int> error{0};
        std::thread helper[kPipeThreads];
        int started = 1;
        // a helper that cannot be started leaves its chunks to be done here afterwards
        for (; started < threads; ++started) {
            try {
                helper[started] = std::thread(work, h, std::cref(chunks), down, started, threads, std::ref(error));
            } catch (...) {   // no thread or no memory for one
                break;
            }
        }
        work(h, chunks, down, 0, threads, error);
        for (int t = 1; t < started; ++t) helper[t].join();
        for (int t = started; t < threads; ++t) work(h, chunks, down, t, threads, error);
        if (error.load()) return failed(h, (cudaError_t)error.load());
    }
    if (down) {
        const cudaError_t e = cudaStreamSynchronize(h->stream);
        if (e != cudaSuccess) return failed(h, e);
    }
    return SLAQ_OK;
}

// The lists of a copy are its only allocations; without memory for them nothing of the caller's may still be in use on return.
int copy_or_fail(slaq_handle* h, Segments segments, bool down) {
    try {
        return copy(h, segments, down);
    } catch (const std::bad_alloc&) {
        cudaStreamSynchronize(h->stream);
        h->err = "out of memory";   // short enough to need none
        return SLAQ_E_NOMEM;
    }
}

}  // namespace

// Ordinary memory that is page-locked afterwards: a third of what cudaHostAlloc takes at the sizes used here (0.3 to 0.5 ms
// against 1.2 to 2.5 ms up to 1 MB).
void* page_locked_alloc(size_t bytes) {
    const size_t size = (bytes + 4095) / 4096 * 4096;
    void* const m = std::aligned_alloc(4096, size);
    void* seen = nullptr;
    if (!m) return nullptr;
    if (cudaHostRegister(m, size, cudaHostRegisterPortable | cudaHostRegisterMapped) == cudaSuccess) {
        if (cudaHostGetDevicePointer(&seen, m, 0) == cudaSuccess && seen == m) return m;   // kernels use the same address
        cudaHostUnregister(m);
    }
    cudaGetLastError();
    std::free(m);
    return nullptr;
}

void page_locked_free(void* m) {
    if (!m) return;
    cudaHostUnregister(m);
    std::free(m);
}

int pipe_to_device(slaq_handle* h, Segments segments) { return copy_or_fail(h, segments, false); }
int pipe_to_host(slaq_handle* h, Segments segments) { return copy_or_fail(h, segments, true); }

void pipe_retain() {
    std::lock_guard<std::mutex> hold(pool().count_lock);
    ++pool().handles;
}

void pipe_release() {
    Pool& p = pool();
    std::lock_guard<std::mutex> hold(p.count_lock);
    if (--p.handles > 0) return;
    std::lock_guard<std::mutex> use(p.lock);
    if (p.memory) page_locked_free(p.memory);
    p.memory = nullptr;
    p.earned = 0;
    p.asked.clear();
    for (const Pool::Spare& s : p.spares) cudaFree(s.memory);
    p.spares.clear();
    for (auto it = p.blocks.begin(); it != p.blocks.end();) {
        if (it->second.taken) {
            ++it;   // freed when it is given back
            continue;
        }
        p.block_bytes -= it->second.bytes;
        page_locked_free(const_cast<char*>(it->first));
        it = p.blocks.erase(it);
    }
}

// A scheduler that takes over from another one makes its call buffer in the middle of its first call, and the driver takes 0.3
// to 20 ms for that; the one it replaces has just given its own back.  At most kSpares buffers and kSpareBytes are kept.
constexpr size_t kSpares = 4, kSpareBytes = 128 << 20;

void* spare_take(int device, size_t bytes, size_t* got) {
    Pool& p = pool();
    std::lock_guard<std::mutex> hold(p.count_lock);
    for (auto it = p.spares.begin(); it != p.spares.end(); ++it) {
        if (it->device != device || it->bytes < bytes) continue;
        void* const memory = it->memory;
        *got = it->bytes;
        p.spares.erase(it);
        return memory;
    }
    return nullptr;
}

void spare_give(int device, void* memory, size_t bytes) {
    Pool& p = pool();
    {
        std::lock_guard<std::mutex> hold(p.count_lock);
        size_t kept = bytes;
        for (const Pool::Spare& s : p.spares) kept += s.bytes;
        if (p.handles > 0 && p.spares.size() < kSpares && kept <= kSpareBytes) {
            try {
                p.spares.push_back({device, memory, bytes});
                return;
            } catch (const std::bad_alloc&) {   // then it is not kept
            }
        }
    }
    cudaFree(memory);
}

bool in_result_block(const void* q, size_t bytes) {
    Pool& p = pool();
    std::lock_guard<std::mutex> hold(p.count_lock);
    const char* const at = static_cast<const char*>(q);
    auto it = p.blocks.upper_bound(at);
    if (it == p.blocks.begin()) return false;
    --it;
    return it->second.taken && at + bytes <= it->first + it->second.bytes;
}

}  // namespace slaq

void* slaq_result_take(size_t bytes) try {
    using namespace slaq;
    size_t size = kResultLeast;
    while (size < bytes) size <<= 1;
    Pool& p = pool();
    std::lock_guard<std::mutex> hold(p.count_lock);
    for (auto& b : p.blocks)
        if (!b.second.taken && b.second.bytes == size) {
            b.second.taken = true;
            return const_cast<char*>(b.first);
        }
    if (p.handles == 0 || size > kResultBytes || ++p.asked[size] <= kResultEarned) return nullptr;
    for (auto it = p.blocks.begin(); it != p.blocks.end() && p.block_bytes + size > kResultBytes;) {   // make room
        if (it->second.taken) {
            ++it;
            continue;
        }
        p.block_bytes -= it->second.bytes;
        page_locked_free(const_cast<char*>(it->first));
        it = p.blocks.erase(it);
    }
    if (p.block_bytes + size > kResultBytes) return nullptr;
    void* const m = page_locked_alloc(size);
    if (!m) return nullptr;
    try {
        p.blocks[static_cast<char*>(m)] = {size, true};
    } catch (const std::bad_alloc&) {
        page_locked_free(m);
        return nullptr;
    }
    p.block_bytes += size;
    return m;
} catch (const std::bad_alloc&) {
    return nullptr;   // the binding takes ordinary memory
}

void slaq_result_give(void* block) {
    using namespace slaq;
    Pool& p = pool();
    std::lock_guard<std::mutex> hold(p.count_lock);
    auto it = p.blocks.find(static_cast<char*>(block));
    if (it == p.blocks.end()) return;
    it->second.taken = false;
    if (p.handles > 0) return;
    p.block_bytes -= it->second.bytes;
    p.blocks.erase(it);
    page_locked_free(block);
}
