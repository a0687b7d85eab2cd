// Barrier over all blocks of a cooperative launch, with a bounded wait.
#pragma once
#include <cuda_runtime.h>

namespace obc {

constexpr int GRID_BARRIER_LIMIT = 1 << 22;       // polls before a block gives up (about a second)

// `arrived` counts arrivals since the launch (zero before it); `target` = gridDim.x times the number of this barrier,
// counted from 1.  Called by every thread of every block; false, for the whole block, when the others did not come in time.
// `limit`: polls (GRID_BARRIER_LIMIT unless a test wants the wait to expire).
__device__ __forceinline__ bool grid_barrier(unsigned int* arrived, unsigned int target, int limit) {
    __syncthreads();
    bool ok = true;
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(arrived, 1u);
        ok = false;
        for (int i = 0; i < limit && !ok; ++i) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
            ok = v >= target;
            if (!ok && i > 256) __nanosleep(64);
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

}  // namespace obc
