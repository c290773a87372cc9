// Grid barrier of the cooperative kernels (SVD sweeps, Lanczos steps): one counter word in global
// memory, zero before the first use.
#pragma once

#include <cuda_runtime.h>

namespace heff {

// about a second: a barrier that has not completed by then never will
constexpr long long GRID_BARRIER_CYCLES = 2ll << 30;

// All threads of nblocks blocks (blockIdx.x < nblocks) meet.  Block 0 adds 2^31 - (nblocks - 1), the
// others 1: the last arrival flips the counter's top bit and leaves the rest zero, so the word serves
// any number of barriers and launches, and a block waits for the bit it saw to change.  An arrival is one
// atomic and the release is that of the last block: with a counter that the last block clears and a
// generation word (three dependent trips to L2 more) a barrier of 152 blocks took 2.1 us.
// Gives up when *err is raised, or after GRID_BARRIER_CYCLES, in which case it raises *err; returns whether
// the blocks met.
__device__ __forceinline__ bool grid_barrier(unsigned int* count, unsigned int nblocks, int* err) {
    __syncthreads();
    __shared__ int ok;
    if (threadIdx.x == 0) {
        ok = 1;
        __threadfence();
        const unsigned int old = atomicAdd(count, blockIdx.x == 0 ? 0x80000000u - (nblocks - 1) : 1u);
        const long long t0 = clock64();
        for (int i = 1; !((old ^ *(volatile unsigned int*)count) & 0x80000000u); ++i) {
            if (i % 8 == 0 && (*(volatile int*)err || clock64() - t0 > GRID_BARRIER_CYCLES)) {
                atomicExch(err, 1);
                ok = 0;
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

}  // namespace heff
