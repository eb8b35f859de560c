// Shared-memory addresses and bounded mbarrier waits.
//
// A wait that runs past its limit returns false; its kernel then counts a
// timeout in a device counter (read and cleared by the host, which reports
// LBM_ETIMEOUT) and returns, so that a missing completion can never hang the GPU.
// No step kernel waits; the self-test (selftest.cu) does.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace lbm {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// makes initialised barriers visible to the asynchronous (TMA) proxy
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}

// Waits for the given phase parity; gives up after about 2^31 clock cycles
// (about one second) and returns false.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < (1ll << 31))
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

}  // namespace lbm
