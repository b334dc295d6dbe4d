// Bulk asynchronous copies into shared memory (PTX cp.async.bulk, completed
// on an mbarrier through its transaction count) and bounded waits on them.
// Every wait gives up at a deadline of the global nanosecond timer, so a
// copy that never lands ends in an error flag instead of a hung kernel.
#pragma once

#include <cstdint>

namespace xdcg {

constexpr unsigned long long kDrainNs = 100000000ull;    // 0.1 s to let copies land

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

// makes initialised barriers visible to the asynchronous (copy) proxy
__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// one arrival that also announces the bytes the phase waits for
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
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

// true once the phase with this parity has completed; false at the deadline.
// The deadline is checked before every try (a try itself may block for a
// while), so a deadline already passed gives up at once, whatever the copy.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          unsigned long long deadline) {
    while (global_ns() < deadline)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// the same for a phase that has usually completed: tried once before the clock is
// read, which costs some 200 cycles (290 per stage of a product at 8^3, of 1900; 1 to
// 1.5 % of a solve).  A warp's first wait is mbar_wait's.
__device__ __forceinline__ bool mbar_wait_next(uint64_t *bar, uint32_t parity,
                                               unsigned long long deadline) {
    return mbar_try_wait(bar, parity) || mbar_wait(bar, parity, deadline);
}

// orders this thread's earlier generic accesses to shared memory before
// later asynchronous-proxy writes (a bulk copy into a buffer just read)
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ uint64_t l2_stream_policy() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// global -> shared bulk copy of `bytes` (multiple of 16, both addresses
// 16-byte aligned), completing on bar
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes,
                                         uint64_t *bar, uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
        "[%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

}  // namespace xdcg
