// host_pages.h -- page-locked host pages for the results of synchronous calls.
#pragma once

#include <cstddef>

#include <cuda_runtime_api.h>

namespace su2 {

// A page of page-locked host memory for the results of a synchronous call:
// copies to it are queued behind the kernels, where a copy to pageable memory
// waits for them (about 8 us each, one after the other).  Pages come from a
// process-wide pool of at most kHostPages, taken for the duration of a call;
// p is NULL when none is free (or page-locking failed), and the call then
// copies to its caller's memory directly.  A call that has synchronised its
// stream after the last copy says so by settled(); otherwise (it returns early,
// on an error) the destructor waits for the stream, so that nothing is on its
// way to a page that the next call takes.
constexpr size_t kHostPageBytes = 64 * 1024;
constexpr int kHostPages = 16;
struct HostPage {
    char *p;
    explicit HostPage(cudaStream_t stream);
    ~HostPage();
    HostPage(const HostPage &) = delete;
    HostPage &operator=(const HostPage &) = delete;
    void settled() { settled_ = true; }

private:
    const cudaStream_t stream_;
    bool settled_ = false;
};

// Every lattice and batch retains the pages while it lives; the last one to go
// gives them back but for kHostPagesKept, which stays with the process.  A
// program that makes a lattice, reads a value and destroys it, again and again,
// would otherwise page-lock and free a page each time: 8^4, us per such turn
// 211 without pages, 542 with all of them given back, 197 so.
constexpr int kHostPagesKept = 1;
void host_pages_retain();
void host_pages_release();

}  // namespace su2
