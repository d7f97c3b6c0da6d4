// When the 8-slice split of an FP64 product is as accurate as an FP64 sum.
//
// A split operand is a fixed-point number relative to its row's (column's) exponent e, so a
// term a_k b_k is off by up to 2^-59 2^(ea+eb), however small it is: 2^-62 2^(ea+eb) from
// the last digits of a and b and 7.03 2^-62 from the pairs of slices that are left out.  An
// FP64 sum is off by up to K u S with u = 2^-53 and S = sum_k |a_k| |b_k|, and by about u S on
// ordinary data.  So what counts is how S / K compares to 2^(ea+eb), for the worst row of A
// with the worst column of B.  The split is taken where S / 2^(ea+eb) is at least 2^-8.2 sqrt(K)
// and 2^-6 for every entry of the product: its error is then at most 4.6 sqrt(K) u S and K u S,
// and on digits that are not all alike about u S / 2.  Two ways to see that:
//   * counts, taken while the operands are cut: for t = 2 .. 8 the most entries of any row that
//     are below 2^(e-t), ma(t) and mb(t).  At least K - ma(t) - mb(v) terms then are above
//     2^(ea-t) 2^(eb-v), and summing over the levels
//       S / 2^(ea+eb) >= sum_{t,v} w_t w_v max(0, K - ma(t) - mb(v)), w_t = 2^-(t+1), w_8 = 2^-8.
//     Gaussian operands pass from K = 28 on (8000 rows: 2^-10.4 K where 2^-10.6 K is needed);
//   * where the counts are too few, the product of the magnitudes' leading 7 bits, one chunk
//     more of every tile (gemm_tc.cu), entry by entry: S / 2^(ea+eb) >= 2^-14 sum_k floor(2^7 |a_k| / 2^ea)
//     floor(2^7 |b_k| / 2^eb).  The contractions and Gram products of a chain pass (by at least a
//     factor of 4 in the cases looked at), operands graded against each other do not.
#pragma once
#include <cuda_runtime.h>

namespace cbc {

constexpr int GUARD_LEVELS = 7;               // t = 2 .. 8
// words of one problem: A's levels, B's levels, an operand holds Inf or NaN, an entry is too
// small; zeroed before the operands are cut
constexpr int GUARD_B = 7, GUARD_BAD = 14, GUARD_FAIL = 15, GUARD_WORDS = 16;
constexpr int GUARD_ZERO_ROW = -4000;         // exponent of a row of zeros (its products are exact)

// K: terms of the real sums (2 K for complex operands)
__device__ __forceinline__ float guard_line(int K) {
  return fmaxf(3.4e-3f * sqrtf((float)K), 0x1p-6f);  // 2^-8.2 sqrt(K)
}
// (not inlined: the roles of a kernel must come to one answer)
static __device__ __noinline__ bool counts_hold(const int* g, int K) {
  float s = 0.f;
#pragma unroll
  for (int t = 0; t < GUARD_LEVELS; ++t) {
    float r = 0.f;
#pragma unroll
    for (int v = 0; v < GUARD_LEVELS; ++v)
      r += (float)max(0, K - g[t] - g[GUARD_B + v]) * (v < 6 ? 0.125f / (1 << v) : 0x1p-8f);
    s += r * (t < 6 ? 0.125f / (1 << t) : 0x1p-8f);
  }
  return s >= guard_line(K);
}
// once the operands are cut and the entries of problems with too few counts are looked at
__device__ __forceinline__ bool split_holds(const int* g) {
  return !g[GUARD_BAD] && !g[GUARD_FAIL];
}

}  // namespace cbc
