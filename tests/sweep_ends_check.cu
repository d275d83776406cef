// Host-side check that the sizes of test_gpu_sweep_units.py take the form it is about on a GPU
// of 152 SMs: with any margin that a level step's box may have (0 to 8 cells, and the whole
// array), sweep_split cuts the double-float columns of at least one axis end to end.
// Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cstdio>

#include "internal.h"

using namespace dfn;

int main() {
  const int sizes[4][3] = {{200, 48, 120}, {64, 160, 96}, {160, 128, 64}, {144, 144, 144}};
  int checks = 0;
  for (const int* n : sizes)
    for (int margin = 0; margin <= 8; ++margin) {
      Box b{};
      for (int d = 0; d < 3; ++d) {
        b.lo[d] = 8 - margin;
        b.hi[d] = 8 + n[d] + margin;
      }
      int ends = 0;
      for (int d = 0; d < 3; ++d) ends += sweep_split(b, d, sweep_blocks(8, d), 152, true) < 0;
      if (!ends) {
        std::printf("FAIL %d %d %d margin %d\n", n[0], n[1], n[2], margin);
        return 1;
      }
      ++checks;
    }
  std::printf("OK %d\n", checks);
  return 0;
}
