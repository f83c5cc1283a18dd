// quotient() against the compiler's division: equal bits for every integer
// divisor, at most the other neighbour for others, equal bits for special values.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include <limits>
#include <random>

#include "quotient.h"

static uint64_t bits(double v) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return b;
}
static double from(uint64_t b) {
  double v;
  std::memcpy(&v, &b, 8);
  return v;
}
static bool same(double a, double b) { return bits(a) == bits(b) || (std::isnan(a) && std::isnan(b)); }

static long bad = 0;
static void check(double x, double d, int far) {
  const double r = 1.0 / d, got = sr::quotient(x, d, r), want = x / d;
  bool ok = same(got, want);
  if (!ok && far)
    ok = std::isfinite(got) && std::isfinite(want) &&
         std::llabs((long long)bits(got) - (long long)bits(want)) <= far;
  if (!ok && bad++ < 10) std::printf("%a / %a: %a, not %a\n", x, d, got, want);
}

int main() {
  std::mt19937_64 rng(5);
  auto value = [&](int lo, int hi) {  // a random sign, significand and exponent
    const uint64_t e = (uint64_t)(1023 + lo + (int)(rng() % (uint64_t)(hi - lo + 1)));
    return from((rng() & 0x800fffffffffffffull) | e << 52);
  };
  for (uint32_t d = 1; d <= 4000; ++d)
    for (int t = 0; t < 300; ++t) check(value(-1022, 1023), d, 0);
  for (int t = 0; t < 1000000; ++t) check(value(-60, 2), (double)(1 + rng() % 0x7fffffffull), 0);
  // products of the divisor and of the neighbours of its multiples
  for (int t = 0; t < 300000; ++t) {
    const double d = (double)(1 + rng() % 0x7fffffffull), m = (double)(rng() % 0x3fffffull) * d;
    for (double x : {m, std::nextafter(m, 1e300), std::nextafter(m, -1e300)}) check(x, d, 0);
  }
  for (int t = 0; t < 1000000; ++t) check(value(-1022, 1023), std::fabs(value(-150, 150)), 1);
  const double inf = std::numeric_limits<double>::infinity();
  for (double d : {1.0, 3.0, 7.0, 2147483647.0, 0.1, 1e-40, 1e30})
    for (double x : {0.0, -0.0, inf, -inf, std::nan(""), 5e-324, -5e-324, 2.2250738585072014e-308,
                     1.7976931348623157e308, -1.7976931348623157e308, 1e-290, 1e290})
      check(x, d, 0);
  std::printf("%ld wrong\n", bad);
  return bad != 0;
}
