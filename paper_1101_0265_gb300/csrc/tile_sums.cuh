// Pieces shared by the products whose tiles are summed as 64-bit integers
// (f64_digits.cu, digits_fixed.cu).
#pragma once

#include <cuda_runtime.h>

#include "digits_kernel.cuh"

namespace purify {

// Launched with programmatic stream serialization: the kernel's prologue runs
// beside its predecessor's tail; memory is touched only after the
// predecessor has completed, and the successor may then start its own prologue.
__device__ __forceinline__ void grid_dependency_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                           Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

namespace dk {

// 8 columns of the four accumulators, 32 lanes each; tmem_wait32 orders the
// registers' use after the loads.
__device__ __forceinline__ void tmem_issue32(uint32_t taddr, uint32_t (&r)[32]) {
#pragma unroll
    for (int a = 0; a < 4; ++a)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[8 * a]), "=r"(r[8 * a + 1]), "=r"(r[8 * a + 2]), "=r"(r[8 * a + 3]),
                       "=r"(r[8 * a + 4]), "=r"(r[8 * a + 5]), "=r"(r[8 * a + 6]), "=r"(r[8 * a + 7])
                     : "r"(taddr + (uint32_t)(a * TILE)));
}

__device__ __forceinline__ void tmem_wait32(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]),
                   "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28])
                 :: "memory");
    asm volatile("" : "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
}

// A float of magnitude below 2^22 plus 1.5 2^23 has its nearest integer in its
// low bits (the conversion instruction runs at 16 per clock and SM).
constexpr float kMagic = 12582912.f;
constexpr unsigned int kMagicBits = 0x4B400000u;

}  // namespace dk
}  // namespace purify
