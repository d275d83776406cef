// Host-side check of transfer_all (hostbuf.h) with transfers that only count: whichever of
// them fails, none follows it, the ones started are waited for once and last, and the first
// code comes back.  Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cstdio>

#include "hostbuf.h"

int main() {
  long long checks = 0;
  for (int n = 0; n <= 60; ++n)
    for (int bad = 0; bad <= n; ++bad)  // bad == n: none fails
      for (int late = 0; late < 2; ++late) {  // late: the wait fails too
        int started = 0, in_flight = 0, waits = 0;
        bool told = false;
        const int rc = dfn::transfer_all(
            n,
            [&](int k) {
              if (k != started || waits) return -99;
              ++started;
              if (k == bad) return -7;
              ++in_flight;
              return 0;
            },
            [&](bool failed) {
              told = failed;
              in_flight = 0;
              ++waits;
              return late ? -3 : 0;
            });
        const int want = bad < n ? -7 : late ? -3 : 0;
        if (rc != want || in_flight || waits != 1 || told != (bad < n) ||
            started != (bad < n ? bad + 1 : n)) {
          std::printf("FAIL n %d bad %d late %d\n", n, bad, late);
          return 1;
        }
        ++checks;
      }
  std::printf("OK %lld\n", checks);
  return 0;
}
