// Helpers of the tensor-core (tcgen05) kernels (tc_gemm.cu, ptc.cu): bounded mbarrier waits,
// shared-memory operand descriptors and tensor-memory set-up.
#pragma once

#include <cstdint>

namespace dlz {

constexpr int kWaitPolls = 1 << 22;     // (each poll may suspend the thread for a while)

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Operand descriptor at shared address `saddr`: 14 address bits (16-byte units) and the
// leading byte offset in the low word, stride byte offset and the descriptor version of the
// sm_100 family (no swizzle) in the high word.  Only the low word changes along K.
__device__ __forceinline__ uint32_t sdesc_lo(uint32_t saddr) { return ((saddr >> 4) & 0x3FFF) | (128u >> 4) << 16; }
template <uint32_t SBO> constexpr uint32_t kDescHi = (SBO >> 4) | 1u << 14;

__device__ __forceinline__ void commit_to(uint64_t *mbar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(mbar)));
}

// Bounded wait for the completion of phase `parity` of an mbarrier.  A wait that gives up
// sets the block's fail word, which ends the other waits as well.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity, volatile int *failed) {
    uint32_t done = 0;
    for (int it = 0; it < kWaitPolls && !done; ++it) {
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}\n"
                     : "=r"(done) : "r"(su32(mbar)), "r"(parity) : "memory");
        if (!done && *failed) return false;
    }
    if (!done) *failed = 1;
    return done != 0;
}
// The issuing warp, before it leaves: waits (lane 0, bounded) until the MMAs it has issued are
// done.  A block gives its tensor and shared memory back after this, also when one of its waits
// has given up and nobody waits for the last MMAs any more.  mbar: one arrival, used only here.
__device__ __forceinline__ void mma_drain(uint64_t *mbar, bool issued, volatile int *failed) {
    if (issued && (threadIdx.x & 31) == 0) {
        commit_to(mbar);
        int none = 0;                      // (not the block's fail word, which ends a wait)
        if (!mbar_wait(mbar, 0, &none)) *failed = 1;
    }
    __syncwarp();
}
__device__ __forceinline__ void mbar_arrive(uint64_t *mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(mbar)) : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t *mbar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(mbar)), "r"(count));
}

// tensor memory of `ncols` columns, allocated by warp 0 into *tbase (all threads call; the
// address is valid after a block barrier and tcgen05.fence::after_thread_sync)
__device__ __forceinline__ void tmem_alloc(uint32_t *tbase, int ncols) {
    if ((threadIdx.x >> 5) == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tbase)), "r"(ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
}

__device__ __forceinline__ void tc_teardown(uint32_t taddr, int ncols) {
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if ((threadIdx.x >> 5) == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}

__device__ __forceinline__ int tmem_cols(int n) { return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512; }

}  // namespace dlz
