// lbm_grid_barrier.cuh -- barrier among the blocks of one cooperative launch,
// with a bounded wait.
#pragma once
#include "lbm_bulk.cuh"

namespace tlv {

constexpr unsigned long long BARRIER_LIMIT_NS = 1000000000ull;

// Every block adds one to *count, which is zero when the launch begins, and
// waits until it reaches `target` (blocks x barriers passed so far). Stores
// made by any block before the barrier are visible after it to loads that go
// past the L1 cache. The whole block calls it; false if the wait ran out
// (the other blocks' waits then run out too, and every block returns).
__device__ __forceinline__ bool grid_barrier(unsigned *count, unsigned target)
{
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        unsigned long long t0 = 0;
        unsigned v, polls = 0;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            if (v >= target) break;
            if ((++polls & 255u) == 0) {  // the clock is read only by waits that are already long
                const unsigned long long t = global_ns();
                if (t0 == 0) {
                    t0 = t;
                } else if (t - t0 > BARRIER_LIMIT_NS) {
                    ok = 0;
                    break;
                }
            }
        }
    }
    return __syncthreads_and(ok) != 0;
}

} // namespace tlv
