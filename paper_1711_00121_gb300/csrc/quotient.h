// Quotients by a divisor whose reciprocal is known.
#pragma once

#include <cmath>
#include <cstdint>

#include "fx64.h"

namespace sr {

// x / d for r = 1 / d rounded to nearest and 2^-150 <= d < 2^150: the product
// q = x r, which is off by less than 1.5 units in its last place, and one
// correction by the remainder x - q d, which an FMA gives exactly (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor",
// 1990).  The error before the last rounding is below 2^-52 units, so the result is
// x / d rounded to nearest unless x / d lies that close to the middle of two
// numbers.  For an integer d below 2^31 it does not: it is at least 2^-32 units
// away.  For another d it may be the other neighbour there.  Results below
// 2^-767, whose remainder could underflow, and those that overflow, infinities and
// NaN take the division; one look at the exponent of the result tells.
FX_HD double quotient_fast(double x, double d, double r) {
  const double q = x * r;
  return fma(fma(-q, d, x), r, q);
}
// +0 or -0, by the two words: as 64 bits the compiler makes it a comparison on the
// FP64 pipe, which the three operations above already fill (5,120 rows of 1,024:
// 42 us, so 32)
FX_HD bool quotient_zero(double c) {
#if defined(__CUDA_ARCH__)
  return ((__double2hiint(c) & 0x7fffffff) | __double2loint(c)) == 0;
#else
  return fx_bits(c) << 1 == 0;
#endif
}
// whether quotient_fast's c is x / d (a zero but for its sign)
FX_HD bool quotient_ok(double c) {
  return (unsigned)(fx_exp(c) - 256) < 1790u || quotient_zero(c);
}
FX_HD double quotient(double x, double d, double r) {
  const double c = quotient_fast(x, d, r);
  return quotient_ok(c) && !quotient_zero(c) ? c : x / d;
}

}  // namespace sr
