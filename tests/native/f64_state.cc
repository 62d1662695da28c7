// Host logic of the float64 digit products (f64_digits.cu) against a stand-in
// for the CUDA runtime: device memory is host memory, a launch only leaves a
// mark in the fixed-point sums, and calls fail when told to.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "f64_digits.h"

static int g_launches, g_fail_launch_at = -1, g_cleared;
static cudaError_t g_copy_error = cudaSuccess;
static unsigned char* g_sums;
static size_t g_sums_bytes;

extern "C" {
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
char __cudaInitModule(void**) { return 0; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t*, const void*) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }

cudaError_t cudaMalloc(void** p, size_t n) {
    *p = malloc(n);
    return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
    if (p == g_sums) g_sums = nullptr;
    free(p);
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
    memset(p, v, n);
    if (n > 64) {  // the sums (the flags are two ints)
        ++g_cleared;
        g_sums = (unsigned char*)p;
        g_sums_bytes = n;
    }
    return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
    if (g_copy_error != cudaSuccess) return g_copy_error;
    memcpy(d, s, n);
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
    *d = 0;
    return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
    *v = 152;
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaPeekAtLastError(void) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) {
    if (g_launches++ == g_fail_launch_at) return cudaErrorLaunchFailure;
    if (g_sums) g_sums[g_sums_bytes - 1] = 1;  // partial sums under way
    return cudaSuccess;
}
}

namespace purify {
int make_quad_map(CUtensorMap*, const __nv_bfloat16*, int) { return PURIFY_OK; }
void count_launches(int) {}
int cuda_status(cudaError_t e, const char*) { return e == cudaErrorMemoryAllocation ? PURIFY_ERR_OOM : PURIFY_ERR_CUDA; }
}  // namespace purify

using namespace purify;

static int g_bad;
#define CHECK(x)                                        \
    do {                                                \
        if (!(x)) {                                     \
            printf("line %d: %s\n", __LINE__, #x);      \
            ++g_bad;                                    \
        }                                               \
    } while (0)

static F64Digits f;
static double X[2], red[4];

static bool begin() {
    int err = 0;
    const bool on = f64d_begin(f, 200, 1, 0, nullptr, &err);
    CHECK(err == PURIFY_OK);
    return on;
}
static int step() { return f64d_step(f, X, X, X, X + 1, 200, 1.0, 0.0, 0.0, 1.0, 0.0, red, nullptr); }
static int check() {
    int redo = 0, flag = 0;
    const int r = f64d_read(f, nullptr);
    return r == PURIFY_OK ? f64d_check(f, &redo, &flag) : r;
}
// The finish pass of a step that ends well clears the sums it has read.
static int good_step_and_check() {
    const int r = step();
    if (r != PURIFY_OK) return r;
    g_sums[g_sums_bytes - 1] = 0;
    return check();
}
static bool sums_are_zero() {
    for (size_t i = 0; i < g_sums_bytes; ++i)
        if (g_sums[i]) return false;
    return true;
}

int main() {
    // a run that ends well leaves the sums zero: the next one does not clear them again
    CHECK(begin() && g_cleared == 1);
    CHECK(good_step_and_check() == PURIFY_OK);
    CHECK(begin() && g_cleared == 1 && sums_are_zero());
    // a step, found complete, then one whose wait runs out
    CHECK(good_step_and_check() == PURIFY_OK);
    CHECK(step() == PURIFY_OK);
    f.flags[1] = 32;
    CHECK(check() == PURIFY_ERR_DEVICE_TIMEOUT);
    CHECK(begin() && sums_are_zero());
    // ... whose finish pass cannot be launched
    CHECK(good_step_and_check() == PURIFY_OK);
    g_fail_launch_at = g_launches + 1;  // the product, then the finish pass (the operand's digits are held)
    CHECK(step() == PURIFY_ERR_CUDA);
    g_fail_launch_at = -1;
    CHECK(begin() && sums_are_zero());
    // ... whose flags cannot be read
    CHECK(good_step_and_check() == PURIFY_OK);
    CHECK(step() == PURIFY_OK);
    g_copy_error = cudaErrorUnknown;
    CHECK(check() == PURIFY_ERR_CUDA);
    g_copy_error = cudaSuccess;
    CHECK(begin() && sums_are_zero());
    // ... that nobody checks
    CHECK(good_step_and_check() == PURIFY_OK);
    CHECK(step() == PURIFY_OK);
    CHECK(begin() && sums_are_zero());
    // an operand that does not fit: checked, and cleared for the next run
    CHECK(step() == PURIFY_OK);
    f.flags[0] = 1;
    int redo = -1, flag = 0;
    CHECK(f64d_check(f, &redo, &flag) == PURIFY_ERR_INTERNAL);  // (not read back yet)
    CHECK(f64d_read(f, nullptr) == PURIFY_OK && f64d_check(f, &redo, &flag) == PURIFY_OK && redo == 0);
    CHECK(begin() && sums_are_zero());
    f64d_free(f);
    printf(g_bad ? "failed\n" : "ok\n");
    return g_bad != 0;
}
