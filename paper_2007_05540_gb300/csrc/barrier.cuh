// Grid barrier of the cooperative kernels (SVD sweeps, Lanczos steps): a counter and a
// generation word in global memory, both zero before the first use.
#pragma once

#include <cuda_runtime.h>

namespace heff {

// about a second: a barrier that has not completed by then never will
constexpr long long GRID_BARRIER_CYCLES = 2ll << 30;

// All threads of nblocks blocks meet.  Gives up when *err is raised, or after
// GRID_BARRIER_CYCLES, in which case it raises *err; returns whether the blocks met.
__device__ __forceinline__ bool grid_barrier(unsigned int* count, unsigned int* gen, unsigned int nblocks,
                                             int* err) {
    __syncthreads();
    __shared__ int ok;
    if (threadIdx.x == 0) {
        ok = 1;
        volatile unsigned int* vgen = gen;
        const unsigned int g = *vgen;
        __threadfence();
        if (atomicAdd(count, 1u) == nblocks - 1) {
            atomicExch(count, 0u);
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            const long long t0 = clock64();
            while (*vgen == g) {
                if (*(volatile int*)err || clock64() - t0 > GRID_BARRIER_CYCLES) {
                    atomicExch(err, 1);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

}  // namespace heff
