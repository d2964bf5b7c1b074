// Bulk asynchronous copies (TMA, cp.async.bulk) and mbarrier helpers for the
// persistent pipelined kernels, plus the device-side error flag their bounded
// waits report to.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bplg {

// Device error word of the including translation unit: 0 = fine; a kernel
// whose bounded wait ran out writes a nonzero code here and returns.  Each
// file that launches pipelined kernels reads and clears its own word for
// bplg_device_status().
static __device__ int g_device_error;

constexpr int kErrWaitTimeout = 1;
// about one second at 2 GHz: far beyond any legitimate copy latency
constexpr long long kWaitLimitCycles = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make mbarrier initialisation visible to the async (TMA) proxy
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// order earlier generic-proxy shared-memory accesses before later async-proxy ones
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// 1-D bulk copy global -> shared, completion counted on `bar` (bytes and both
// addresses must be multiples of 16).
__device__ __forceinline__ void tma_load_1d(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
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

// Wait for phase `parity` of `bar` with a time limit; false (and the device
// error word set) if the limit passed.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  long long limit = kWaitLimitCycles) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) {
            atomicExch(&g_device_error, kErrWaitTimeout);
            return false;
        }
    }
    return true;
}

// The same by every thread of a block with one phase in flight, which leaves when
// the vote on it fails.  The leader waits twice as long, so when the vote fails the
// copies have been waited for again and have landed, or that has run out too: the
// shared memory may belong to another block afterwards.  (A wait after the vote
// does the same, but its code in the loop cost the bulk-copy tridiagonal solver 4 us
// of 60 at n = 3000.)
__device__ __forceinline__ bool mbar_wait_block(uint64_t *bar, uint32_t parity, bool leader) {
    return mbar_wait_bounded(bar, parity, leader ? 2 * kWaitLimitCycles : kWaitLimitCycles);
}

}  // namespace bplg
