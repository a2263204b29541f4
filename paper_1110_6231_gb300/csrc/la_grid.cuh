// Barrier of a co-resident grid (a cooperative launch): arrivals are counted
// on one word in L2 and a generation word releases the waiters.
#pragma once

#include "la.h"
#include "la_device.cuh"

namespace la {

struct GridBar {
    unsigned arrived;
    unsigned generation;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Every thread of every CTA calls it; writes before it are visible to reads
// after it. A wait longer than 2 s sets LA_ERR_INTERNAL in *status and
// returns false (in all threads of the CTA) instead of spinning on; *s_ok is
// a shared word of the CTA that starts at 1. The waiter polls without
// sleeping: a barrier of 152 CTAs then costs about as much as two L2 round
// trips, and a sleep's granularity would be most of a barrier's time.
__device__ __forceinline__ bool grid_barrier(GridBar *bar, int *status, int *s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned g = ld_acquire_u32(&bar->generation);
        __threadfence();
        if (atomicAdd(&bar->arrived, 1u) + 1 == gridDim.x) {
            atomicExch(&bar->arrived, 0u);
            __threadfence();
            atomicAdd(&bar->generation, 1u);
        } else {
            const unsigned long long t0 = global_timer_ns();
            for (unsigned it = 1; ld_acquire_u32(&bar->generation) == g; ++it) {
                if ((it & 63u) == 0 && global_timer_ns() - t0 > 2000000000ull) {
                    atomicCAS(status, 0, (int)LA_ERR_INTERNAL);
                    *s_ok = 0;
                    break;
                }
            }
        }
        __threadfence();
    }
    __syncthreads();
    return *s_ok != 0;
}

}  // namespace la
