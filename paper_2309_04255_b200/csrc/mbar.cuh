// Shared-memory barriers (mbarrier) and the election of an issuing lane, for the kernels that feed the
// tensor cores.
#pragma once

#include "common.cuh"

namespace llmcad {

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait of a warp whose lanes stay together (the MMA warps): every lane tries, so that no broadcast follows.
__device__ __forceinline__ bool mbar_wait_all(uint32_t bar, uint32_t parity, volatile int *abort_flag, uint64_t wait_limit)
{
    uint64_t t0 = 0;
    for (uint32_t it = 1; !__all_sync(0xffffffffu, mbar_try(bar, parity)); ++it) {
        if ((it & 255u) == 0) {
            bool out = *abort_flag != 0;
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            else out |= now - t0 > wait_limit;
            if (__any_sync(0xffffffffu, out)) return false;
        }
    }
    return true;
}
// Whether the phase is complete, without waiting.
__device__ __forceinline__ bool mbar_test_all(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return __all_sync(0xffffffffu, ok != 0);
}
// The same for two barriers at once.
__device__ __forceinline__ bool mbar_test2_all(uint32_t bar_a, uint32_t parity_a, uint32_t bar_b, uint32_t parity_b)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 q, [%3], %4;\n\t"
        "and.pred p, p, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar_a), "r"(parity_a), "r"(bar_b), "r"(parity_b)
        : "memory");
    return __all_sync(0xffffffffu, ok != 0);
}
// Threads that issue MMAs: the code between two of them is what limits the rate (one lane under `if (lane == 0)` got
// through 8 MMAs, their commit and two barrier waits in 1250 cycles, four times what the tensor pipe needs for 64
// columns: every operand went through a per-thread register). The MMA warps therefore stay converged, so that
// addresses and descriptors live in uniform registers, and one elected lane issues.
__device__ __forceinline__ bool elect_one()
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)::"memory");
    return ok != 0;
}

}  // namespace llmcad
