// Grid barrier of the cooperative kernels (all blocks resident): arrivals are
// counted in the control block, every wait is bounded, and the last block to
// leave the kernel resets the count.
#pragma once
#include "common.cuh"
#include "grid_count.h"

namespace espp {

constexpr int GRID_WAIT = 1 << 21;  // polls before giving up (a second or so)

// Barrier number `phase` (1, 2, ..) of this launch, called by every thread of
// every block; false if the wait ran out (the error is recorded; the block is to
// leave).  Writes before it are visible to plain loads after it.  after(): run by
// thread 0 between the wait and the block's release.  fault: a barrier of the launch
// whose wait runs out at once, whoever arrives (0: none; the tests' injection).
template <class F>
__device__ __forceinline__ bool grid_barrier(Ctrl* c, unsigned int phase, unsigned int fault, F&& after) {
    __shared__ int arrived;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        const bool never = fault != 0 && phase == fault;
        const unsigned int goal = barrier_goal(gridDim.x, phase) + (never ? 1u : 0u);
        const int limit = never ? 64 : GRID_WAIT;
        atomicAdd(&c->bar, 1u);
        unsigned int seen = 0;
        int it = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&c->bar) : "memory");
        } while (!barrier_reached(seen, goal) && ++it < limit);
        __threadfence();
        after();
        arrived = barrier_reached(seen, goal);
        if (!arrived) {
            atomicOr(&c->err, ERRBIT_TIMEOUT);
            c->abort = 1;
        }
    }
    __syncthreads();
    return arrived != 0;
}

// The end of a kernel with barriers: last() runs in one thread, after every block
// has passed its last barrier.
template <class F>
__device__ __forceinline__ void grid_leave(Ctrl* c, F&& last) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&c->blocks_done, 1u) == gridDim.x - 1) {
            __threadfence();
            c->bar = 0;
            c->blocks_done = 0;
            last();
        }
    }
}

}  // namespace espp
