// Bulk (TMA) copies into shared memory with mbarrier completion, sm_103a
// inline PTX: the 1-D cp.async.bulk form (no tensor map), one issuing thread,
// the copy engine tracking completion by bytes on a shared-memory mbarrier.
#pragma once

#include <stdint.h>

namespace adc {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(unsigned long long *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Global -> shared bulk copy; addresses 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, unsigned long long *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// Bounded wait for the phase of the given parity (polls with a short sleep
// between them, so waiting warps leave the shared-memory pipe to the others);
// false if the limit ran out.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long *bar, uint32_t parity, long long limit) {
    long long it = 0;
    while (!mbar_try_wait(bar, parity)) {
        if (++it > limit) return false;
        __nanosleep(32);
    }
    return true;
}

// The wait of a block that gives up for its own copy in flight: a copy that
// lands after the block has left would write into another block's shared
// memory.  Its limit is its own, since the one that ran out may be short.
constexpr long long kDrainLimit = 1ll << 22;
__device__ __forceinline__ void mbar_drain(unsigned long long *bar, uint32_t parity) {
    mbar_wait_bounded(bar, parity, kDrainLimit);
}

// Orders this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (bulk copy) accesses: issued before refilling a buffer
// that threads have just read.
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

}  // namespace adc
