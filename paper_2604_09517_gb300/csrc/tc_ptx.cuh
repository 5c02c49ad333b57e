// Helpers shared by the tensor-core kernels: mbarriers with bounded waits, proxy
// and tcgen05 fences, commits, operand descriptors, and the fixed-point form of
// an FP64 value that the sliced products cut up.
#pragma once
#include "common.cuh"

namespace hplgb {
namespace tc {

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
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

// Bounded wait. Returns false (and raises the CTA's abort flag and the global
// error word) when the deadline passes or another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t deadline, volatile int* abort,
                                          int* err) {
    while (!mbar_try_wait(bar, parity)) {
        if (*abort) return false;
        if (globaltimer_ns() > deadline) {
            *abort = 1;
            atomicExch(err, HPL_ERR_TIMEOUT);
            return false;
        }
    }
    return true;
}

// generic-proxy writes to shared memory become visible to the async proxy (TMA, tcgen05.mma)
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory descriptor of a K-major tile without swizzle (8 rows x 16
// bytes core matrices): lead bytes between the two k octets, stride bytes
// between groups of 8 rows.
__device__ __forceinline__ uint64_t desc_plain(uint32_t saddr, uint32_t lead, uint32_t stride) {
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | (uint64_t)(lead >> 4) << 16 | (uint64_t)(stride >> 4) << 32 |
           (uint64_t)1 << 46;
}

__device__ __forceinline__ int expo(double v) { return (int)((unsigned)(__double2hiint(v)) >> 20) & 0x7ff; }

// 64-bit fixed point, truncated, of |v| 2^x relative to 2^e (|v| 2^x < 2^e):
// bit 63 has weight 2^(e-1)
__device__ __forceinline__ unsigned long long fixed64(double v, int x, int e) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const int E = (int)(u >> 52) & 0x7ff;
    const unsigned long long m = E ? (u << 11) | (1ull << 63) : 0ull;
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(m), "r"(1022 + e - E - x));    // >= 64: zero
    return r;
}

}  // namespace tc
}  // namespace hplgb
