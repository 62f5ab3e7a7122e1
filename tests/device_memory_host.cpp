// Host build of csrc/device_memory.cpp for tests/test_device_memory_host.py, with a stand-in for
// the CUDA allocator: a device of `g_limit` bytes that counts what is allocated on it.
#include <cstdlib>
#include <mutex>
#include <string>

#include "dlz_internal.cuh"

namespace {
std::mutex g_mu;
size_t g_limit = 0, g_used = 0;
}

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_used + n > g_limit) return cudaErrorMemoryAllocation;
    g_used += n;
    size_t *q = static_cast<size_t *>(std::malloc(sizeof(size_t)));
    *q = n;
    *p = q;
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    std::lock_guard<std::mutex> lk(g_mu);
    g_used -= *static_cast<size_t *>(p);
    std::free(p);
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "stand-in"; }
}

namespace dlz {
int fail(int code, const std::string &) { return code; }
}

using namespace dlz;

extern "C" {
void dm_limit(size_t bytes) { g_limit = bytes; }
size_t dm_used() { return g_used; }
void *dm_pool_new() { return new ScratchPool(); }
void dm_pool_delete(void *p) { delete static_cast<ScratchPool *>(p); }
void *dm_take(void *pool, size_t bytes, int *rc) { return static_cast<ScratchPool *>(pool)->take(bytes, *rc); }
size_t dm_bytes(void *buf) { return static_cast<DevBuf *>(buf)->bytes; }
void dm_give(void *pool, void *buf) { static_cast<ScratchPool *>(pool)->give(static_cast<DevBuf *>(buf)); }
// a plain allocation of the library, freed at once
int dm_alloc(size_t bytes) {
    DevBuf b;
    return b.alloc(bytes);
}
// takes and gives `n` times, writing a mark of this call into the buffer meanwhile; the number of
// times another call's mark was found
int dm_hammer(void *pool, size_t bytes, int n, int mark) {
    int bad = 0;
    for (int i = 0; i < n; ++i) {
        int rc = 0;
        DevBuf *b = static_cast<ScratchPool *>(pool)->take(bytes + (size_t)(i % 7), rc);
        if (!b) return -1;
        size_t *q = static_cast<size_t *>(b->p);
        const size_t size = *q;
        *q = size + ((size_t)mark << 48);
        for (volatile int k = 0; k < 50; ++k) {}
        if (*q >> 48 != (size_t)mark) ++bad;
        *q = size;
        static_cast<ScratchPool *>(pool)->give(b);
    }
    return bad;
}
}
