// pic_wait.cuh -- bounded waits on mbarriers.
//
// A wait on an mbarrier never spins without a limit: it polls up to a time
// budget (globaltimer, nanoseconds) and reports failure.
#pragma once

#include <cstdint>

#include "pic_internal.cuh"

namespace pic {

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// true once the phase with the given parity has completed; false after the
// time budget (from t0) is spent
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t t0, uint64_t budget_ns)
{
    const uint32_t a = smem_addr(bar);
    for (;;) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (global_ns() - t0 > budget_ns) return false;
    }
}

}  // namespace pic
