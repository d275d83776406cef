// Host-side check of the quotient by a sum that cancels (div_sum, df64.h) against long
// double: q = n / (a + b), by a factor of cancellation up to 2^20.
//   The sum is within 2^-46 (|a| + |b|) of a + b, the quotient by it within 2^-42 (df64.h),
// so |q - n / (a + b)| <= |n / (a + b)| (2^-42 + 2^-45 (|a| + |b|) / |a + b|): linear in the
// cancellation (2^-45: the second-order terms are below the first).
// Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cmath>
#include <cstdint>
#include <cstdio>

#include "df64.h"

using namespace dfn;

static uint64_t rng = 0x9e3779b97f4a7c15ull;
static double uniform() {  // xorshift64*, [0, 1)
  rng ^= rng >> 12;
  rng ^= rng << 25;
  rng ^= rng >> 27;
  return (double)((rng * 0x2545f4914f6cdd1dull) >> 11) * 0x1.0p-53;
}
static long double val(df64 v) { return (long double)v.hi + (long double)v.lo; }

int main() {
  long long n = 0;
  for (int k = 0; k < 2000000; ++k) {
    // a background and a deviation that leaves between 2 and 2^-20 of it
    const double a0 = std::pow(10.0, -3.0 + 6.0 * uniform());
    const double left = std::pow(2.0, 1.0 - 21.0 * uniform());
    const df64 a = to_df64(a0), b = to_df64(a0 * (left - 1.0));
    const df64 c = to_df64((uniform() - 0.5) * std::pow(10.0, -3.0 + 6.0 * uniform()));
    const long double S = val(a) + val(b), Q = val(c) / S;
    const long double M = std::fabs(val(a)) + std::fabs(val(b));
    const long double bound = std::fabs(Q) * (0x1.0p-42L + 0x1.0p-45L * M / std::fabs(S));
    if (std::fabs(val(div_sum(c, a, b)) - Q) > bound) {
      std::printf("FAIL %.17g %.17g %.17g\n", (double)val(a), (double)val(b), (double)val(c));
      return 1;
    }
    ++n;
  }
  std::printf("OK %lld\n", n);
  return 0;
}
