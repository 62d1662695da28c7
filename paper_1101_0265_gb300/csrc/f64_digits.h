// Float64 steps on the tensor cores: exact digit products (f64_digits.cu).
#pragma once

#include <cuda_bf16.h>

#include "internal.h"

namespace purify {

// Device buffers of a handle's float64 digit products: up to kF64KeepBytes are kept
// from run to run (and grow with the size), larger ones (at most 2^15 rows: 39
// GB) are given back when a run has ended.  The digits of a step's operands are kept for the run's
// next steps and forgotten at the next f64d_begin.
struct F64Digits {
    int n_pad = 0, cap_pad = 0, ctas = 0;
    __nv_bfloat16* planes[2] = {nullptr, nullptr};
    int* exps[2] = {nullptr, nullptr};  // row exponents of planes[b]
    unsigned long long* T = nullptr;    // fixed-point product, upper 128 x 128 tiles; zero between steps
    bool clean = false;                 // T is zero (every step queued so far was checked and ended well)
    int* flags = nullptr;  // [0] the step (from 1) whose operand left the digits' range; [1] a wait that ran out
    int* host_flags = nullptr;  // (pinned) their copy that f64d_read queued
    bool read = false;          // ... since the last step
    void* rows = nullptr;  // row scales for f64d_test_entries
    const double* held[2] = {nullptr, nullptr};  // the run's matrix whose digits planes[b] hold
    int step = 0;                                // steps queued since f64d_begin
    long long wait_cycles = 0;                   // bound of the products' work waits
};

// Sizes that take the digit products (see f64_digits.cu).
bool f64d_wanted(int64_t n);

// Buffers for size n with the planes of `operands` (1 or 2) matrices, and a
// cleared state for a new run's steps.  False when the size does not want
// them or the device has no room (the caller then takes launch_step_f64); *err
// receives other failures.
bool f64d_begin(F64Digits& f, int64_t n, int operands, long long wait_cycles, cudaStream_t s, int* err);

// MMA flops of one step's product.
double f64d_flops(int64_t n);

// launch_step_f64 by exact digit products (red[2] is not reduced); A, B and E are
// exactly symmetric.
int f64d_step(F64Digits& f, const double* A, const double* B, const double* E, double* C, int64_t n, double cP,
              double cE, double cI, double dY, double dI, double* red, cudaStream_t s);

// Queue a test of the run's result D (F: the run's Hamiltonian): where an entry of
// a product of its rows would be known worse from digits than from a chain of
// FMAs, f64d_check reports it as a step that cannot be held.
int f64d_test_entries(F64Digits& f, const double* D, const double* F, int64_t n, cudaStream_t s);

// Queue the read-back of the steps' flags.
int f64d_read(F64Digits& f, cudaStream_t s);
// After a synchronisation behind f64d_read: the step (from 0) whose operand cannot
// be held, so that it has to be taken with launch_step_f64 (-1: none; that step
// and all later ones have written nothing).  PURIFY_ERR_DEVICE_TIMEOUT and
// *wait_flag != 0 when a device wait ran out.
int f64d_check(F64Digits& f, int* redo_from, int* wait_flag);

// After a run: keep the buffers, or free them when they are large.
void f64d_end(F64Digits& f);
void f64d_free(F64Digits& f);

}  // namespace purify
