// Bulk copies between ordinary host memory and the device.
#pragma once

#include <cstddef>
#include <initializer_list>

struct slaq_handle;

namespace slaq {

struct Segment {
    void* dst;
    const void* src;
    size_t bytes;
};

// Copy all segments, queued on the handle's stream.  to_device: the copies may still run on return, and page-locked sources of
// kPipeFrom bytes and more may still be read by them: the caller waits for the stream before its own caller gets them back.
// to_host: returns once everything has arrived.  Returns 0, or a status with the handle's message set.
struct Segments {
    const Segment* at;
    size_t n;
    Segments(std::initializer_list<Segment> list) : at(list.begin()), n(list.size()) {}
    Segments(const Segment* first, size_t count) : at(first), n(count) {}
    const Segment* begin() const { return at; }
    const Segment* end() const { return at + n; }
};
int pipe_to_device(slaq_handle* h, Segments segments);
int pipe_to_host(slaq_handle* h, Segments segments);

// A handle begins / ends its life: the page-locked buffers behind the copies are shared by all handles of the process
// and released with the last of them.
void pipe_retain();
void pipe_release();

// Page-locked memory at the same address for host and device; null if there is none to be had.
void* page_locked_alloc(size_t bytes);
void page_locked_free(void* m);

// Whether [p, p + bytes) lies in a block handed out by slaq_result_take.
bool in_result_block(const void* p, size_t bytes);

// Device memory that passes from one handle of a device to the next (its last work is done): null where none is large enough.
void* spare_take(int device, size_t bytes, size_t* got);
void spare_give(int device, void* memory, size_t bytes);

}  // namespace slaq

// Page-locked memory for results the binding hands to its caller: the device writes them where they are read, and memory
// that is used again has its pages.  At most 64 MB at a time, in blocks of a power of two; NULL beyond that (the binding
// then takes ordinary memory).  A block that is given back is kept for the next call until the last handle ends.
extern "C" void* slaq_result_take(size_t bytes);
extern "C" void slaq_result_give(void* block);
