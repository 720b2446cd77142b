// Barrier over all CTAs of a cooperative launch, with a poll limit.
#pragma once

#include "common.cuh"

namespace uncomp {

constexpr unsigned kGridBarrierSpin = 1u << 22;

// `bar` counts arrivals monotonically and must be zero when the kernel starts; `phase` is the caller's count of
// barriers passed.  Returns false (and raises UNCOMP_STATUS_TIMEOUT) when the others do not arrive: every CTA then leaves.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned &phase, uint32_t *status, int *flag) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
        const unsigned target = (phase + 1u) * gridDim.x;
        bool ok = false;
        for (unsigned it = 0; it < kGridBarrierSpin; ++it) {
            unsigned cur;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(cur) : "l"(bar) : "memory");
            if (cur >= target) { ok = true; break; }
        }
        if (!ok) atomicOr(status, (uint32_t)UNCOMP_STATUS_TIMEOUT);
        *flag = ok ? 1 : 0;
    }
    __syncthreads();
    ++phase;
    return *flag != 0;
}

}  // namespace uncomp
