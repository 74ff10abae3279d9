// Barrier between all blocks of a cooperative launch (the persistent producers).
#pragma once

#include "asd_internal.h"

namespace asd {

constexpr unsigned long long kGridTimeoutNs = 4000000000ull;

// Barrier over all blocks of a cooperative launch: the count reaches `target` once every
// block has arrived.  The release before the arrival and the acquire after the wait order
// all blocks' global stores and loads around it (the acquire also drops this SM's L1 lines).
// Bounded: false for every thread of the block after kGridTimeoutNs.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned target, int *err)
{
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        __threadfence();
        asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
        unsigned long long t0 = 0;
        for (unsigned it = 0;; ++it) {
            unsigned v;
            asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if ((int)(v - target) >= 0) break;
            if ((it & 1023u) == 1023u) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                else if (now - t0 > kGridTimeoutNs) {
                    atomicCAS(err, 0, (int)DEV_TIMEOUT_GRID);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

}  // namespace asd
