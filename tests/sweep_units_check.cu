// Host-side check of how a fused sweep is cut into units (sweep_unit, sweep_split in
// internal.h) by brute force: over boxes of many shapes, the three directions and both
// forms, every plane of every column belongs to exactly one unit, no unit is empty, and a
// split never asks for fewer planes a unit than its least.
// Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cstdio>
#include <vector>

#include "internal.h"

using namespace dfn;

int main() {
  long long n = 0, ends = 0;
  const int sizes[] = {1, 2, 5, 16, 31, 40, 73, 104, 137, 144};
  for (int d = 0; d < 3; ++d)
    for (int nx : sizes)
      for (int nr : sizes)
        for (int nm : sizes) {
          Box b{};
          for (int k = 0; k < 3; ++k) b.lo[k] = 3;
          const int mu = sweep_march_axis(d);
          b.hi[0] = 3 + nx;
          b.hi[sweep_row_axis(d)] = 3 + nr;
          b.hi[mu] = 3 + nm;
          const int ncol = sweep_columns(b, d);
          const int cuts[] = {1, nm, (nm + 2) / 3, -1, -2, -nm, -nm - 3, -(nm + 2) / 2 - 1,
                              sweep_split(b, d, 3, 152, true), sweep_split(b, d, 7, 152, false)};
          for (int zc : cuts) {
            b.zc = zc;
            std::vector<int> seen((size_t)ncol * nm, 0);
            for (int u = 0; u < sweep_units(b, d); ++u) {
              int pos, end;
              sweep_unit(b, d, u, pos, end);
              if (pos < 0 || end <= pos || end > ncol * nm) {
                std::printf("FAIL unit d %d %d %d %d zc %d: %d\n", d, nx, nr, nm, zc, u);
                return 1;
              }
              for (; pos < end; ++pos) ++seen[pos];
              ++n;
            }
            for (int s : seen)
              if (s != 1) {
                std::printf("FAIL cover d %d %d %d %d zc %d\n", d, nx, nr, nm, zc);
                return 1;
              }
          }
          const int zc = sweep_split(b, d, 4, 152, true), least = d == 0 ? 1 : 4;
          if (zc < 0 ? -zc < least : zc < (nm < least ? nm : least) || zc > nm) {
            std::printf("FAIL split d %d %d %d %d: %d\n", d, nx, nr, nm, zc);
            return 1;
          }
          ends += zc < 0;
        }
  if (!ends) {  // the sizes above hold both forms
    std::printf("FAIL no box takes the columns laid end to end\n");
    return 1;
  }
  std::printf("OK %lld\n", n);
  return 0;
}
