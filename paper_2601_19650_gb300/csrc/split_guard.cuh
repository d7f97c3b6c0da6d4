// When the 8-slice split of an FP64 product is as accurate as an FP64 sum.
//
// A split operand is a fixed-point number relative to its row's (column's) exponent e, so a
// term a_k b_k is off by up to 2^-59 2^(ea+eb), however small it is: 2^-62 2^(ea+eb) from
// the last digits of a and b and 7.03 2^-62 from the pairs of slices that are left out.  An
// FP64 sum is off by up to K u S with u = 2^-53 and S = sum_k |a_k| |b_k|, and by about u S on
// ordinary data.  So what counts is how S / K compares to 2^(ea+eb).  The split is taken where
// S / 2^(ea+eb) is at least 2^-8.2 sqrt(K) and 2^-6 for every entry of the product: its error is
// then at most 4.6 sqrt(K) u S and K u S, and on digits that are not all alike about u S / 2.
// S is bounded from below by the product of the magnitudes' leading 7 bits (gemm_tc.cu, one chunk
// more of every tile):
//   S / 2^(ea+eb) >= 2^-14 sum_k floor(2^7 |a_k| / 2^ea) floor(2^7 |b_k| / 2^eb).
// Gaussian operands are a factor of 2^3.5 to 2^6 above the line, the contractions and Gram
// products of an FP64 application by at least 4 (but for a few whose operands are graded); operands
// graded against each other along K are below it.
#pragma once
#include <cuda_runtime.h>

namespace cbc {

// words of one problem, zeroed before the operands are cut: an operand holds Inf or NaN; an entry
// is below the line
constexpr int GUARD_BAD = 0, GUARD_FAIL = 1, GUARD_WORDS = 2;
constexpr int GUARD_ZERO_ROW = -4000;  // exponent of a row of zeros (its products are exact)

// K: terms of the real sums (2 K for complex operands)
__device__ __forceinline__ float guard_line(int K) {
  return fmaxf(3.4e-3f * sqrtf((float)K), 0x1p-6f);  // 2^-8.2 sqrt(K)
}
// once the tensor-core kernel has been through the problem
__device__ __forceinline__ bool split_holds(const int* g) {
  return !g[GUARD_BAD] && !g[GUARD_FAIL];
}

}  // namespace cbc
