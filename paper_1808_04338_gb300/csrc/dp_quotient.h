// The quotients of a column by one divisor.  On GB300 an FP64 division is some
// twenty instructions that each hold a quarter of the SM for 64 cycles; with
// the divisor's reciprocal at hand a quotient takes three, as accurate.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace dp {

// a / d rounded to nearest, with r = 1 / d rounded to nearest; 0 for d = 0.
// P. Markstein (Computation of elementary functions on the IBM RISC
// System/6000 processor, IBM J. Res. Dev. 34, 1990): the product q = a r, its
// remainder a - q d by one fused operation, and q corrected by it.  The product
// alone has a second rounding (up to 1.5 units in the last place).  Where the
// reciprocal, the quotient or the remainder might leave the normal range
// (|.| below 2^-900 or from 2^900 on, infinities, NaN) it is the division.
#ifdef __CUDACC__
__host__ __device__
#endif
inline double quotient(double a, double d, double r) {
  auto bits = [](double v) {
    uint64_t b;
    memcpy(&b, &v, sizeof b);
    return b;
  };
  auto mid = [&](double v) {   // 2^-900 <= |v| < 2^900
    return ((uint32_t)(bits(v) >> 52) & 0x7ffu) - (1023u - 900u) < 1800u;
  };
  const double q = a * r;
  if (mid(d)) {
    if (mid(a) && mid(q)) return fma(fma(-q, d, a), r, q);
    if ((bits(a) << 1) == 0) return q;
  } else if ((bits(d) << 1) == 0) {
    return 0.0;
  }
  return a / d;
}

}  // namespace dp
