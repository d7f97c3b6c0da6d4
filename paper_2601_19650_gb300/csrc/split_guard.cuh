// When the 8-slice split of an FP64 product is as accurate as an FP64 sum.
//
// A split operand is a fixed-point number relative to its row's (column's) exponent e, so a
// term a_k b_k is off by up to 2^-59 2^(ea+eb), however small it is: 2^-62 2^(ea+eb) from
// the last digits of a and b and 7.03 2^-62 from the pairs of slices that are left out.  An
// FP64 sum is off by up to K u S with u = 2^-53 and S = sum_k |a_k| |b_k|, and by about u S on
// ordinary data.  So what counts is how S / K compares to 2^(ea+eb), for the worst row of A
// with the worst column of B.  Counted while the operands are cut: for t = 2 .. 8 the most
// entries of any row that are below 2^(e-t), ma(t) and mb(t).  At least K - ma(t) - mb(v)
// terms then are above 2^(ea-t) 2^(eb-v), and summing over the levels
//   S / 2^(ea+eb) >= sum_{t,v} w_t w_v max(0, K - ma(t) - mb(v)),  w_t = 2^-(t+1), w_8 = 2^-8.
// The split is taken where that is at least 2^-8.2 sqrt(K): its error is then at most
// 4.6 sqrt(K) u S, below K u S for K >= 22, and on digits that are not all alike about u S / 2.
// Gaussian operands pass from K = 28 on (8000 rows: 2^-10.4 K, and 2^-10.6 K is needed; K = 20
// fails); operands graded along K, or with many zeros, and Inf or NaN do not.
#pragma once
#include <cuda_runtime.h>

namespace cbc {

constexpr int GUARD_LEVELS = 7;               // t = 2 .. 8
constexpr int GUARD_B = 7, GUARD_BAD = 14;    // words: A's levels, B's levels, Inf or NaN
constexpr int GUARD_WORDS = 16;               // of one problem, zeroed before the operands are cut

// K: terms of the real sums (2 K for complex operands)
__device__ __forceinline__ bool split_holds(const int* g, int K) {
  if (g[GUARD_BAD]) return false;
  float s = 0.f;
#pragma unroll
  for (int t = 0; t < GUARD_LEVELS; ++t) {
    float r = 0.f;
#pragma unroll
    for (int v = 0; v < GUARD_LEVELS; ++v)
      r += (float)max(0, K - g[t] - g[GUARD_B + v]) * (v < 6 ? 0.125f / (1 << v) : 0x1p-8f);
    s += r * (t < 6 ? 0.125f / (1 << t) : 0x1p-8f);
  }
  return s >= 3.4e-3f * sqrtf((float)K);  // 2^-8.2
}

}  // namespace cbc
