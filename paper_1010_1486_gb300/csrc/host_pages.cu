// host_pages.cu -- the pool of page-locked result pages.  Host code on CUDA's
// runtime interface alone.
#include <mutex>

#include "host_pages.h"

namespace su2 {

static std::mutex g_page_mutex;
static char *g_pages[kHostPages];  // the free ones
static int g_pages_free = 0, g_pages_made = 0, g_page_users = 0;

HostPage::HostPage(cudaStream_t stream) : p(nullptr), stream_(stream)
{
    std::lock_guard<std::mutex> lock(g_page_mutex);
    if (g_pages_free > 0) {
        p = g_pages[--g_pages_free];
    } else if (g_pages_made < kHostPages) {
        void *q = nullptr;
        if (cudaHostAlloc(&q, kHostPageBytes, cudaHostAllocPortable) == cudaSuccess) {
            p = (char *)q;
            ++g_pages_made;
        } else {
            cudaGetLastError();
        }
    }
}

HostPage::~HostPage()
{
    if (!p) return;
    if (!settled_ && cudaStreamSynchronize(stream_) != cudaSuccess) cudaGetLastError();
    std::lock_guard<std::mutex> lock(g_page_mutex);
    g_pages[g_pages_free++] = p;
}

void host_pages_retain()
{
    std::lock_guard<std::mutex> lock(g_page_mutex);
    if (++g_page_users > 1) return;
    // the pages kept while there was no handle: still there unless the program reset the device
    for (int i = g_pages_free; i-- > 0;) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, g_pages[i]) == cudaSuccess && at.type == cudaMemoryTypeHost) continue;
        g_pages[i] = g_pages[--g_pages_free];
        --g_pages_made;
    }
    cudaGetLastError();
}

void host_pages_release()
{
    std::lock_guard<std::mutex> lock(g_page_mutex);
    if (--g_page_users > 0) return;
    while (g_pages_free > kHostPagesKept) {
        cudaFreeHost(g_pages[--g_pages_free]);
        --g_pages_made;
    }
    cudaGetLastError();
}

}  // namespace su2
