// Grid-wide barrier of a cooperative launch, with a bounded wait.
#pragma once

#include <cuda_runtime.h>

namespace ewv {

__device__ __forceinline__ unsigned long long grid_now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Barrier over all blocks: bar[0] counts arrivals over the launch (zero before it), `phase` counts
// the barriers of this launch from 1.  Each wait lasts at most limit_ns.  Returns false (in every
// thread of the block) if it gave up.  What a block wrote before the barrier is visible to every
// block after it: thread 0's release and acquire at gpu scope cover the block's other threads
// through the block barriers around them (a fence in every thread costs microseconds).
__device__ __forceinline__ bool grid_phase_barrier(unsigned int* bar, unsigned int phase, unsigned long long limit_ns,
                                                   int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        const unsigned int want = phase * gridDim.x;
        bool ok = true;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        const unsigned long long t0 = grid_now_ns();
        for (unsigned int it = 1;; ++it) {
            unsigned int seen;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
            if (seen >= want) break;
            // (a limit of zero, for testing: only a barrier that all have reached passes)
            if (limit_ns == 0 || ((it & 63u) == 0 && grid_now_ns() - t0 > limit_ns)) {
                ok = false;
                break;
            }
        }
        *s_ok = ok ? 1 : 0;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Leaving a launch that used the barrier: the last block clears bar[0] and bar[1] for the next one.
__device__ __forceinline__ void chain_leave(unsigned int* bar) {
    __syncthreads();
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        __threadfence();
        if (atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
            bar[0] = 0u;
            bar[1] = 0u;
            __threadfence();
        }
    }
}

}  // namespace ewv
