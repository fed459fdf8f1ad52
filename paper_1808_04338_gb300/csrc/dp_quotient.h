// The quotients of a column by one divisor.  On GB300 an FP64 division is some
// twenty instructions that each hold a quarter of the SM for 64 cycles; with
// the divisor's reciprocal at hand a quotient takes three, as accurate.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace dp {

#ifdef __CUDACC__
#define DP_QUOTIENT __host__ __device__ __forceinline__
#else
#define DP_QUOTIENT inline
#endif

// Tests of a double by its bits (an FP64 comparison is an FP64 instruction too).
DP_QUOTIENT uint64_t quotient_bits(double v) {
  uint64_t b;
  memcpy(&b, &v, sizeof b);
  return b;
}
DP_QUOTIENT bool quotient_mid(double v) {   // 2^-900 <= |v| < 2^900
  return ((uint32_t)(quotient_bits(v) >> 52) & 0x7ffu) - (1023u - 900u) < 1800u;
}
DP_QUOTIENT bool quotient_zero(double v) { return (quotient_bits(v) << 1) == 0; }

// a / d rounded to nearest, with r = 1 / d rounded to nearest, when *ok.
// P. Markstein (Computation of elementary functions on the IBM RISC
// System/6000 processor, IBM J. Res. Dev. 34, 1990): the product q = a r, its
// remainder a - q d by one fused operation, and q corrected by it.  The product
// alone has a second rounding (up to 1.5 units in the last place).  Not *ok
// where the reciprocal, the quotient or the remainder might leave the normal
// range (|.| below 2^-900 or from 2^900 on, infinities, NaN).  No branches, so
// that several quotients overlap.
DP_QUOTIENT double quotient_if(double a, double d, double r, bool *ok) {
  const double q = a * r, l = fma(fma(-q, d, a), r, q);
  const bool zero = quotient_zero(a);
  *ok = quotient_mid(d) & (zero | (quotient_mid(a) & quotient_mid(q)));
  return zero ? q : l;
}

// a / d, or 0 for d = 0 (as a zero pivot's multipliers are).
DP_QUOTIENT double quotient(double a, double d, double r) {
  bool ok;
  const double l = quotient_if(a, d, r, &ok);
  return ok ? l : quotient_zero(d) ? 0.0 : a / d;
}

}  // namespace dp
