// k_tanh64.cuh -- binary64 tanh for the fused kernels.
//
// A kernel with a binary64 tanh is bound by the FP64 pipe, and CUDA's tanh
// takes 14 of its operations.  This one takes 7: the interval of |x| comes
// from its exponent and leading mantissa bits (integer work), its table row
// holds a node a and tanh's Taylor coefficients at a, and
//   tanh|x| = c0 + h (c1 + h (c2 + ... + h c6)),  h = |x| - a,
// with h exact (Sterbenz).  16 intervals per binade from 2^-9 to 2^-3, 64 up
// to 1 and 128 up to 20 keep the first dropped term, c7 h^7, below 2^-55 of
// the result.  The nodes are Gal's (k_tanh64_table.cuh): tanh(a) lies within
// 2^-12 ulp of the stored c0, so the error is the final rounding plus less
// than 0.1 ulp.  Below 2^-9 the row is the series at 0, and from 20 on tanh
// rounds to 1.
//
// Measured: at most 0.57 ulp from 2^-9 on and 1 ulp below (host build of this
// source against 120-bit values).  On a GB300 the 20-step reverse pass of a
// 256^3 binary64 tanh chain, whose 20 forward steps evaluate it once per
// cell, went from 19.4 to 15.2 ms.
#include "k_tanh64_table.cuh"

__device__ __forceinline__ double dcp_tanh64(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned long long m = b & 0x7fffffffffffffffull;
  const unsigned hi = (unsigned)(m >> 32);
  if (hi >= 0x40340000u)  // |x| >= 20, NaN
    return m > 0x7ff0000000000000ull
               ? x
               : __longlong_as_double((long long)((b ^ m) | 0x3ff0000000000000ull));
  unsigned i = 0;
  if (hi >= 0x3f600000u) i = 1u + ((hi - 0x3f600000u) >> 16);
  if (hi >= 0x3fc00000u) i = 97u + ((hi - 0x3fc00000u) >> 14);
  if (hi >= 0x3ff00000u) i = 289u + ((hi - 0x3ff00000u) >> 13);
  const double2* row = reinterpret_cast<const double2*>(dcp_tanh_tab[i]);
  const double2 r0 = __ldg(row), r1 = __ldg(row + 1), r2 = __ldg(row + 2), r3 = __ldg(row + 3);
  const double h = __dsub_rn(__longlong_as_double((long long)m), r0.x);
  double p = __fma_rn(h, r3.y, r3.x);
  p = __fma_rn(h, p, r2.y);
  p = __fma_rn(h, p, r2.x);
  p = __fma_rn(h, p, r1.y);
  p = __fma_rn(h, p, r1.x);
  p = __fma_rn(h, p, r0.y);
  return __longlong_as_double((long long)((b ^ m) | (unsigned long long)__double_as_longlong(p)));
}
