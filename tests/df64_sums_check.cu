// Host-side check of the unnormalised double-float sums (add_u, sub_u, fsub_u, norm;
// df64.h) against FP64, over operands that cancel to every degree:
//   s = a + b            |s - (a + b)| <= 2^-46 (|a| + |b|), |lo| <= 2^-22 (|a| + |b|)
//   s c, s / c           the sum's error times c (over c), and 2^-46 (|a| + |b|) |c|
//                        (2^-42 |s / c| + 2^-44 (|a| + |b|) / |c|)
//   s + c                2^-45 (|a| + |b| + |c|)
//   norm(s)              the same value, |lo| <= half an ulp of hi
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
static double operand() {
  const double mag = std::pow(10.0, -6.0 + 8.0 * uniform());
  return (uniform() < 0.5 ? -1.0 : 1.0) * mag * (1.0 + uniform());
}
static double val(df64 v) { return (double)v.hi + (double)v.lo; }

int main() {
  long long n = 0;
  for (int k = 0; k < 2000000; ++k) {
    const double x = operand();
    // half of the pairs nearly cancel, by a factor down to 2^-44
    const double y = k & 1 ? operand() : -x * (1.0 + std::pow(2.0, -44.0 * uniform()));
    const df64 a = to_df64(x), b = to_df64(y), c = to_df64(operand());
    const double A = val(a), B = val(b), C = val(c), M = std::fabs(A) + std::fabs(B);
    const df64 s = k % 3 == 0 ? add_u(a, b) : k % 3 == 1 ? sub_u(a, -b) : fsub_u(a.hi, -b);
    const double S = k % 3 == 2 ? (double)a.hi + B : A + B;
    const df64 q = norm(s);
    if (std::fabs(val(s) - S) > 0x1.0p-46 * M || std::fabs(s.lo) > 0x1.0p-22 * M ||
        std::fabs(val(mul_u(s, c)) - S * C) > 0x1.0p-44 * M * std::fabs(C) ||
        std::fabs(val(div_u(s, c)) - S / C) >
            0x1.0p-42 * std::fabs(S / C) + 0x1.0p-44 * M / std::fabs(C) ||
        std::fabs(val(s + c) - (S + C)) > 0x1.0p-45 * (M + std::fabs(C)) ||
        val(q) != val(s) || q.hi + q.lo != q.hi) {
      std::printf("FAIL %.17g %.17g %.17g\n", A, B, C);
      return 1;
    }
    ++n;
  }
  std::printf("OK %lld\n", n);
  return 0;
}
