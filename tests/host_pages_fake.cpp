// The page pool (host_pages.cu) over a fake of the runtime calls it makes.
// Each scenario prints one line of what it saw.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "host_pages.cu"

static int n_alloc = 0, n_free = 0, n_sync = 0, live = 0;
static cudaStream_t last_sync = nullptr;

extern "C" {
cudaError_t cudaHostAlloc(void **p, size_t bytes, unsigned int)
{
    ++n_alloc;
    ++live;
    *p = malloc(bytes);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p)
{
    ++n_free;
    --live;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes *at, const void *)
{
    at->type = live > 0 ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s)
{
    ++n_sync;
    last_sync = s;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
}

using namespace su2;

int main(int argc, char **argv)
{
    const char *what = argc > 1 ? argv[1] : "";
    cudaStream_t a = (cudaStream_t)0x10, b = (cudaStream_t)0x20;
    if (!strcmp(what, "settle")) {
        host_pages_retain();
        {
            HostPage p(a);
            p.settled();
        }
        printf("%d ", n_sync);  // a call that synchronised does not wait again
        {
            HostPage p(b);  // returns early, as on an error
        }
        printf("%d %d ", n_sync, last_sync == b);
        {
            std::vector<HostPage *> all;
            for (int i = 0; i < kHostPages + 1; ++i) all.push_back(new HostPage(a));
            printf("%d ", all.back()->p == nullptr);  // the pool is bounded
            n_sync = 0;
            for (HostPage *p : all) delete p;
            printf("%d ", n_sync);  // none for the call without a page
        }
        host_pages_release();
        printf("%d\n", n_alloc);
    }
    if (!strcmp(what, "turns")) {
        for (int turn = 0; turn < 5; ++turn) {
            host_pages_retain();
            HostPage *p[3];
            for (HostPage *&q : p) (q = new HostPage(a))->settled();
            for (HostPage *q : p) delete q;
            host_pages_release();
        }
        printf("%d %d %d ", n_alloc, n_free, live);
        live = 0;  // the program resets the device: the page kept is gone
        host_pages_retain();
        {
            HostPage p(a);
            p.settled();
        }
        printf("%d %d ", n_alloc, n_free);
        host_pages_release();
        printf("%d %d\n", n_free, live);
    }
    return 0;
}
