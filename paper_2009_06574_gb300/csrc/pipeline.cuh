// Shared-memory barriers (inline PTX, sm_90+) of the drawing pass. Every wait is
// bounded.
#pragma once
#include <stdint.h>

namespace hexfc {

#ifndef HEXFC_WAIT_CYCLES
#define HEXFC_WAIT_CYCLES (1ll << 30)
#endif
constexpr long long kWaitCycles = HEXFC_WAIT_CYCLES;   // about half a second of SM clock (a build-time choice, for tests)

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// Make barrier initialisation visible to the other threads and to the async proxy.
__device__ __forceinline__ void mbar_init_fence()
{
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_addr(bar)) : "memory");
}
// Whether the phase with parity `parity` has completed (does not wait).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, unsigned parity)
{
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

}  // namespace hexfc
