// Bounded grid-wide barrier for cooperative launches (every block resident).
#pragma once

#include <cuda_runtime.h>

// Each block's thread 0 adds one to a counter (a release reduction, no answer awaited) that is never
// reset, and polls it with acquire loads until it reaches the block count times the number of
// barriers so far, which every block counts for itself.  The counter's top bit says that some wait
// gave up, so the polled word carries the outcome too.  A barrier is then one trip to the L2 for
// the arrival and one observed poll after the last one.  101 thin solves of 67 level steps took 38 ms
// with a generation word read before an atomic arrival and released by the last block, and an error
// word read after it; 35.8 with one counter and a line of its own to poll; 32.5 with the counter alone.
// The counter must be zero at the launch; 2^31 / blocks barriers fit a launch.  The wait is bounded:
// `limit` counts units of 64 ns of the global timer (200,000 ~ 13 ms, 20,000,000 ~ 1.3 s); a block
// whose wait runs out records a timeout, and every block leaves the kernel at its next barrier.
struct GridBar {
    unsigned int count;      // arrivals since the launch; kGridFailed
    int pad0[31];
    int err;                 // for the host, on a line of its own
    int pad1[31];
};
constexpr unsigned int kGridFailed = 0x80000000u;

__device__ __forceinline__ unsigned int gb_ld_acquire(const unsigned int *p) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void gb_arrive(unsigned int *p) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}

__device__ __forceinline__ unsigned long long gb_clock_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// every block leaves at its next barrier, the host reads err
__device__ __forceinline__ void grid_fail(GridBar *bar) {
    atomicExch(&bar->err, 1);
    atomicOr(&bar->count, kGridFailed);
}

// The thread that arrives and polls: in the last warp, which the first items of small steps leave idle.
__device__ __forceinline__ bool grid_speaker() { return threadIdx.x == blockDim.x - 32; }

// The barrier in two halves, for work between them that neither reads what other blocks write
// before the barrier nor writes what they read: every thread calls both.  `at` is the block's count
// of arrivals to wait for, zero before the first barrier.
__device__ __forceinline__ void grid_arrive(GridBar *bar, unsigned int nblocks, unsigned int &at) {
    __syncthreads();
    if (grid_speaker()) gb_arrive(&bar->count);
    at += nblocks;
}

__device__ __forceinline__ bool grid_wait(GridBar *bar, long long limit, unsigned int at) {
    __shared__ int s_ok;     // one outcome per block, read by all of its threads
    if (grid_speaker()) {
        unsigned long long deadline = 0;
        unsigned int polls = 0, v = gb_ld_acquire(&bar->count);
        while (v < at) {     // kGridFailed makes v large
            if ((++polls & 63u) == 0u) {
                const unsigned long long now = gb_clock_ns();
                if (deadline == 0) deadline = now + 64ull * (unsigned long long)limit;
                if (now > deadline) {
                    grid_fail(bar);
                    v = kGridFailed;
                    break;
                }
            }
            v = gb_ld_acquire(&bar->count);
        }
        s_ok = !(v & kGridFailed);
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ __forceinline__ bool grid_barrier(GridBar *bar, unsigned int nblocks, long long limit, unsigned int &at) {
    grid_arrive(bar, nblocks, at);
    return grid_wait(bar, limit, at);
}
