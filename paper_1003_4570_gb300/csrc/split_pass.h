// Passes of a restart's many-output combination (combine_split_kernel in lanczos.cu).
#pragma once

#include <algorithm>

#include "smem.cuh"

// A pass of combine_split_kernel: `cols` columns by the kernel of `kernel` >= cols.
struct SplitPass {
  int cols, kernel;
};
// The pass that begins with `left` of `total` columns to go, from na vectors.  25 columns a pass where
// that saves passes over 16 (49 of a basis of 96: two, not four; 32 of a basis of 64 stay at two of 16),
// and what is left at the end goes to the narrowest kernel that holds it: a pass costs its kernel's
// columns (its vectors are read once, and every product is formed).  The coefficients of a pass stay
// in shared memory, so long bases take narrower ones.  400 steps at 640k rows: basis 64 (32 columns)
// 99.0 ms with two passes of 25, 95.6 ms with two of 16; basis 128 (64) 148.7 ms with three of 25,
// 147.1 ms with 25, 25, 16; basis 96 (48 and 49) 121 ms, twice 25, either way.
inline SplitPass split_pass(int na, int total, int left) {
  auto fits = [&](int cols) { return (size_t)na * cols * sizeof(float2) <= kMaxDynamicSmem; };
  const int most = (total + 24) / 25 < (total + 15) / 16 && fits(25) ? 25 : fits(16) ? 16 : 8;
  const int cols = std::min(most, left);
  return SplitPass{cols, cols <= 8 ? 8 : cols <= 16 ? 16 : 25};
}
