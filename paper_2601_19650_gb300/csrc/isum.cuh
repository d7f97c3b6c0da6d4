// Sums over a CTA in integers, for the reductions to tridiagonal form: no FP64 instruction
// (~64 clocks each on this part) and the same value in every CTA that adds the same terms.
#pragma once
#include <cuda_runtime.h>

namespace cbc {

// Exact sums of up to 256 doubles in 64-bit integers.  A term m 2^(e-1075) (m of 53 bits)
// enters as m 2^2 shifted right by its distance to the largest exponent, rounded, so what is
// lost is below 2^-55 of the largest term.
struct WarpSum {
  long long sum;
  int e;  // exponent field of the largest term
};
__device__ __forceinline__ WarpSum warp_isum(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffu);
  const int emax = __reduce_max_sync(0xffffffffu, e);
  const unsigned long long m = e ? ((b & 0xfffffffffffffull) | (1ull << 52)) << 2 : 0ull;
  const int sh = emax - e;
  unsigned long long q = 0ull;
  if (sh == 0)
    q = m;
  else if (sh < 60)
    q = (m + (1ull << (sh - 1))) >> sh;
  // three limbs (26, 26 and the rest) through the 32-bit warp reduction
  const long long s = (b >> 63) ? -(long long)q : (long long)q;
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)s & 0x3ffffffu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(s >> 26) & 0x3ffffffu);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(s >> 52));
  return {((long long)hi << 52) + ((long long)mid << 26) + (long long)lo, emax};
}
// total of the warps' sums, rounded to a double
template <int NW>
__device__ __forceinline__ double block_isum(const WarpSum* s) {
  int E = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) E = max(E, s[w].e);
  long long t = 0;
#pragma unroll
  for (int w = 0; w < NW; ++w) t += s[w].sum >> min(E - s[w].e, 63);
  if (E == 0x7ff) return __longlong_as_double(0x7ff8000000000000LL);  // a NaN or Inf among them
  if (t == 0) return 0.0;
  const unsigned long long neg = t < 0 ? 1ull : 0ull;
  unsigned long long m = neg ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int top = 63 - __clzll((long long)m);
  int ex = E + top - 54;  // the term 2^54 of a sum has the exponent field E
  if (top > 52) {
    const int sh = top - 52;
    m = (m + (1ull << (sh - 1))) >> sh;
    if (m >> 53) {
      m >>= 1;
      ++ex;
    }
  } else {
    m <<= 52 - top;
  }
  if (ex <= 0) return 0.0;
  if (ex >= 0x7ff) return __longlong_as_double(0x7ff0000000000000LL);
  return __longlong_as_double(
      (long long)((neg << 63) | ((unsigned long long)ex << 52) | (m & 0xfffffffffffffull)));
}

}  // namespace cbc
