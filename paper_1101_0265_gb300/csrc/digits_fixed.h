// Digit-plane products with fixed-point sums and a separate finish pass
// (digits_fixed.cu).
#pragma once

#include "digits_tc.h"

namespace purify {

// Whether a step takes this path: dense, 7-bit remainder digits, less than two
// waves of tiles, its buffers given (DigitStep::fixed).
bool digits_fixed_wanted(const DigitStep& st);
bool digits_fixed_size(int n_pad, int ctas);

// Buffers for products of up to `tiles` tiles (0.5 MB for one, 70 MB at the end of
// this path's range on 152 SMs) and their release.
int alloc_fixed_sums(int tiles, int ctas, FixedSums* f);
void free_fixed_sums(FixedSums* f);

// Make that path's kernels ready (once per process; call before capturing
// launches into a graph).
int prepare_digit_fixed();

// launch_digit_step by that path (two launches).
int launch_digit_fixed(const DigitStep& st, cudaStream_t stream);

}  // namespace purify
