// Grid-wide barrier of a cooperative launch, with a bounded wait.
#pragma once

#include "tfsph_internal.cuh"

namespace tfsph {

struct GridBar {
    unsigned int count;
    unsigned int gen;
};

__device__ __forceinline__ unsigned int ld_acquire(const unsigned int *p)
{
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// The last CTA to arrive resets the count and advances the generation; the
// others wait for the generation to change, at most spin_limit clock cycles.
// Returns false (after flagging kErrTimeout) when the wait ran out; the
// caller then returns at once.
__device__ __forceinline__ bool grid_barrier(GridBar *bar, long long spin_limit, int *err, unsigned int sleep_ns)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const unsigned int g = ld_acquire(&bar->gen);
        __threadfence();
        if (atomicAdd(&bar->count, 1u) == gridDim.x - 1) {
            atomicExch(&bar->count, 0u);
            __threadfence();
            atomicAdd(&bar->gen, 1u);
        } else {
            const long long t0 = clock64();
            while (ld_acquire(&bar->gen) == g) {
                if (clock64() - t0 > spin_limit) {
                    atomicOr(err, kErrTimeout);
                    ok = 0;
                    break;
                }
                if (sleep_ns) __nanosleep(sleep_ns);
            }
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

}  // namespace tfsph
