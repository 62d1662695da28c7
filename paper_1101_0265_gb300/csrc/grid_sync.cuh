// A bounded grid-wide barrier for cooperative launches.
#pragma once

#include <cuda_runtime.h>

namespace purify {

// Words of a barrier in device memory, zero at launch: arrivals, and a flag set
// when a wait ran out: every later wait then returns at once, the kernel runs to
// its end, and its caller does the work again launch by launch. (Blocks of
// another stream's kernel may hold SMs for longer than any bound while part of
// the grid already waits.)
struct GridSync {
    unsigned int arrived, failed;
};

// Every thread of every block calls it the same number of times; `round` counts
// the calls.  All blocks are resident (cooperative launch).  `limit`: clocks one
// wait may take (0: about one second).
__device__ __forceinline__ void grid_barrier(GridSync* g, unsigned int& round, long long limit) {
    ++round;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&g->arrived, 1u);
        const unsigned int need = round * gridDim.x;
        const long long t0 = clock64();
        unsigned int v;
        for (;;) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&g->arrived) : "memory");
            if (v >= need || *(volatile unsigned int*)&g->failed) break;
            if (clock64() - t0 > (limit > 0 ? limit : 1ll << 31)) {
                *(volatile unsigned int*)&g->failed = 1u;
                break;
            }
        }
        __threadfence();
    }
    __syncthreads();
}

}  // namespace purify
