// Signed 64-bit fixed point on the device's integer pipe: conversions from and
// to floating point, and the product with a reciprocal.  GB300 issues FP64
// instructions, and conversions from or to 64-bit types, at 1/64 of the FP32
// rate; sums of such integers are exact.
#pragma once

#include "sr_internal.h"

namespace sr {

// m * 2^sh rounded to nearest (half away from zero), negated when neg
__device__ __forceinline__ long long fixed_shift(uint64_t m, int sh, bool neg) {
  long long f = 0;
  if (sh >= 0)
    f = (long long)(m << sh);
  else if (sh > -60)
    f = (long long)((m + (1ull << (-sh - 1))) >> -sh);
  return neg ? -f : f;
}

// v * 2^(56 - e) for |v| < 2^e
__device__ __forceinline__ long long fixed_of(float v, int e) {
  const uint32_t b = __float_as_uint(v);
  const int x = (int)((b >> 23) & 0xffu);
  const uint32_t m = x ? (b & 0x7fffffu) | 0x800000u : b & 0x7fffffu;
  return fixed_shift(m, max(x, 1) - 150 + 56 - e, (b >> 31) != 0);
}
__device__ __forceinline__ long long fixed_of(double v, int e) {
  const uint64_t b = (uint64_t)__double_as_longlong(v);
  const int x = (int)((b >> 52) & 0x7ffu);
  const uint64_t m = x ? (b & 0xfffffffffffffull) | 0x10000000000000ull : b & 0xfffffffffffffull;
  return fixed_shift(m, max(x, 1) - 1075 + 56 - e, (b >> 63) != 0);
}

// out of line: instructions that a launch runs once are bound by their fetch
static __device__ __noinline__ double fixed_value_slow(long long v, int e) {
  return ldexp((double)v, e);
}

// v * 2^e rounded to nearest even; ODD (FP32): rounded to odd instead, for a
// second rounding to fewer bits
template <typename T, bool ODD = false>
__device__ __forceinline__ T fixed_value(long long v, int e) {
  if (v == 0) return T(0);
  const uint64_t a = v < 0 ? (uint64_t)-v : (uint64_t)v;
  const int lz = __clzll((long long)a);
  const int x = 63 - lz + e;  // 2^x <= |v| 2^e
  constexpr bool F = sizeof(T) == 4;
  if (x < (F ? -126 : -1022) || x > (F ? 126 : 1022)) return (T)fixed_value_slow(v, e);
  const uint64_t m = a << lz;
  constexpr int DROP = F ? 40 : 11;
  const uint64_t rem = m & ((1ull << DROP) - 1), half = 1ull << (DROP - 1);
  uint64_t q = m >> DROP;  // leading one included
  if (ODD)
    q |= rem ? 1 : 0;
  else
    q += (rem > half || (rem == half && (q & 1))) ? 1 : 0;
  // adding the significand with its leading one carries into the exponent
  if constexpr (F)
    return __uint_as_float((((uint32_t)(x + 126) << 23) + (uint32_t)q) |
                           (v < 0 ? 0x80000000u : 0u));
  else
    return __longlong_as_double((long long)((((uint64_t)(x + 1022) << 52) + q) |
                                            (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// s times the factor f = r 2^-(63 + s'), f.sh = s' + f.h - 1, rounded to
// nearest; |s| 2^(f.h) < 2^63
__device__ __forceinline__ long long fixed_scale(long long s, const SweepScale& f) {
  const long long t = __mul64hi(s << f.h, (long long)f.r);
  return (t + (1ll << (f.sh - 1))) >> f.sh;
}

// |v| as an FP32 value not below it
__device__ __forceinline__ float up_abs(float v) { return fabsf(v); }
__device__ __forceinline__ float up_abs(double v) { return __double2float_ru(fabs(v)); }

}  // namespace sr
