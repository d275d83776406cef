// Host-side check of the fused sweeps' lane layout (sweep_lane, internal.h) by brute
// force: over boxes of many shapes and the three directions, every cell of the box is
// owned by exactly one lane of the warps of its blocks, the lanes around it hold the
// neighbours its stencil takes by shuffle, and no lane lies outside the box and its halo.
// Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cstdio>
#include <vector>

#include "internal.h"

using namespace dfn;

int main() {
  long long n = 0;
  const int sizes[] = {1, 2, 7, 26, 27, 28, 31, 32, 33, 61, 64, 93, 137};
  for (int d = 0; d < 3; ++d)
    for (int nx : sizes)
      for (int nr : sizes) {
        Box b{};
        const int ra = sweep_row_axis(d), lo = d == 0 ? 3 : 1, hi = d == 0 ? 2 : 0;
        for (int k = 0; k < 3; ++k) {
          b.lo[k] = 5;
          b.hi[k] = 9;
        }
        b.hi[0] = 5 + nx;
        b.hi[ra] = 5 + nr;
        std::vector<int> seen((size_t)nx * nr, 0);
        const int warps = sweep_columns(b, d) * (kSweepThreads / 32);
        for (int w = 0; w < warps; ++w) {
          SweepLane p[32];
          if (!sweep_lane(b, d, w, 0, p[0])) continue;
          for (int l = 0; l < 32; ++l) {
            if (!sweep_lane(b, d, w, l, p[l]) || p[l].x < b.lo[0] - lo ||
                p[l].x >= b.hi[0] + hi || p[l].row < b.lo[ra] || p[l].row >= b.hi[ra]) {
              std::printf("FAIL range d %d nx %d nr %d warp %d lane %d\n", d, nx, nr, w, l);
              return 1;
            }
            ++n;
          }
          for (int l = 0; l < 32; ++l) {
            if (!p[l].mine || p[l].x < b.lo[0] || p[l].x >= b.hi[0]) continue;
            ++seen[(size_t)(p[l].row - b.lo[ra]) * nx + p[l].x - b.lo[0]];
            for (int k = -lo; k <= hi; ++k)
              if (l + k < 0 || l + k > 31 || p[l + k].x != p[l].x + k ||
                  p[l + k].row != p[l].row) {
                std::printf("FAIL neighbour d %d nx %d nr %d warp %d lane %d\n", d, nx, nr, w, l);
                return 1;
              }
          }
        }
        for (int s : seen)
          if (s != 1) {
            std::printf("FAIL cover d %d nx %d nr %d: %d\n", d, nx, nr, s);
            return 1;
          }
      }
  std::printf("OK %lld\n", n);
  return 0;
}
