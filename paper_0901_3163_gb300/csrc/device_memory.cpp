// Device buffers and the work memory that operators keep between calls (dlz_internal.cuh).
#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "dlz_internal.cuh"

namespace dlz {

namespace {
// Every operator's pool, what they hold idle, and the lock of all of them (takes and gives are
// a few per call).  Never destroyed: operators may outlive the library's static objects.
struct Pools {
    std::mutex mu;
    std::vector<ScratchPool *> all;
    size_t idle_bytes = 0;
};
Pools &pools() {
    static Pools *p = new Pools();
    return *p;
}
}  // namespace

int DevBuf::alloc(size_t nbytes) {
    release();
    if (nbytes == 0) return DLZ_OK;
    cudaError_t e = cudaMalloc(&p, nbytes);
    if (e == cudaErrorMemoryAllocation && ScratchPool::free_idle()) {
        cudaGetLastError();
        e = cudaMalloc(&p, nbytes);
    }
    if (e != cudaSuccess) {
        p = nullptr;
        cudaGetLastError();
        return fail(e == cudaErrorMemoryAllocation ? DLZ_ERR_OOM : DLZ_ERR_CUDA,
                    "cudaMalloc(" + std::to_string(nbytes) + "): " + cudaGetErrorString(e));
    }
    bytes = nbytes;
    return DLZ_OK;
}
void DevBuf::release() {
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
}

ScratchPool::ScratchPool() {
    idle.reserve(kKeep);
    std::lock_guard<std::mutex> lk(pools().mu);
    pools().all.push_back(this);
}
ScratchPool::~ScratchPool() {
    std::lock_guard<std::mutex> lk(pools().mu);
    auto &all = pools().all;
    all.erase(std::find(all.begin(), all.end(), this));
    for (DevBuf *b : idle) {
        pools().idle_bytes -= b->bytes;
        delete b;
    }
}
DevBuf *ScratchPool::take(size_t bytes, int &rc) {
    {
        std::lock_guard<std::mutex> lk(pools().mu);
        int best = -1;
        for (int i = 0; i < (int)idle.size(); ++i)
            if (idle[i]->bytes >= bytes && (best < 0 || idle[i]->bytes < idle[best]->bytes)) best = i;
        if (best >= 0) {
            DevBuf *b = idle[best];
            idle.erase(idle.begin() + best);
            pools().idle_bytes -= b->bytes;
            rc = DLZ_OK;
            return b;
        }
    }
    DevBuf *b = new DevBuf();
    rc = b->alloc(bytes);
    if (rc != DLZ_OK) {
        delete b;
        return nullptr;
    }
    return b;
}
void ScratchPool::give(DevBuf *b) {
    if (b->bytes <= kKeepBytes) {
        Pools &ps = pools();
        std::lock_guard<std::mutex> lk(ps.mu);
        const bool full = (int)idle.size() >= kKeep;
        // a full pool gives up its smallest buffer for a larger one
        auto it = std::min_element(idle.begin(), idle.end(), [](DevBuf *x, DevBuf *y) { return x->bytes < y->bytes; });
        const size_t old = full ? (*it)->bytes : 0;
        if (b->bytes > old && ps.idle_bytes - old + b->bytes <= kKeepAllBytes) {
            ps.idle_bytes += b->bytes - old;
            if (full) {
                std::swap(*it, b);
            } else {
                idle.push_back(b);
                return;
            }
        }
    }
    delete b;
}
bool ScratchPool::free_idle() {
    std::lock_guard<std::mutex> lk(pools().mu);
    bool any = false;
    for (ScratchPool *p : pools().all) {
        for (DevBuf *b : p->idle) {
            delete b;
            any = true;
        }
        p->idle.clear();
    }
    pools().idle_bytes = 0;
    return any;
}

}  // namespace dlz
