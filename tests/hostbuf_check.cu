// Host-side check of which host buffers a kernel may reach itself (reachable, hostbuf.h),
// against a map of the pages that are registered: random registrations of an address range,
// side by side and with holes between them, some read-only, some at another distance on the
// device.  Prints "OK <checks>" and exits 0, or the first failure and exits 1.
#include <cstdio>
#include <cstdlib>

#include "hostbuf.h"

using namespace dfn;

int main() {
  constexpr int kUnits = 64;  // of 512 bytes
  constexpr uintptr_t kHost = 0x10000, kUnit = 512;
  std::srand(7);
  long long n = 0, yes = 0, joined = 0;
  for (int round = 0; round < 200000; ++round) {
    // the registration of every unit (-1: none), and what each is
    int owner[kUnits], first[kUnits], units[kUnits], count = 0;
    bool ro[kUnits];
    uintptr_t shift[kUnits];  // device address - host address
    const bool apart = std::rand() % 2;
    for (int u = 0; u < kUnits;) {
      const int len = 1 + std::rand() % 32, end = u + len < kUnits ? u + len : kUnits;
      const bool hole = std::rand() % 4 == 0;
      first[count] = u;
      units[count] = end - u;
      ro[count] = std::rand() % 4 == 0;
      shift[count] = apart && std::rand() % 2 ? 0x7000000 : 0;
      for (; u < end; ++u) owner[u] = hole ? -1 : count;
      if (!hole) ++count;
    }
    const size_t at = 8 * (std::rand() % (kUnits * kUnit / 8));
    const size_t bytes = 8 * (1 + std::rand() % (kUnits * kUnit / 8));
    const bool write = std::rand() % 2;
    auto ask = [&](uintptr_t host) {
      HostPart p = {};
      const uintptr_t off = host - kHost;
      const int o = off < kUnits * kUnit ? owner[off / kUnit] : -1;
      if (o < 0) return p;
      p.pinned = true;
      p.writable = write && !ro[o];
      p.dev = host + shift[o];
      p.start = kHost + shift[o] + first[o] * kUnit;
      p.size = units[o] * kUnit;
      return p;
    };
    // every byte registered, written only where it may be, at one distance on the device
    bool want = true;
    for (size_t b = at; b < at + bytes && want; b += 8) {
      const int o = b < kUnits * kUnit ? owner[b / kUnit] : -1;
      want = o >= 0 && !(write && ro[o]) && shift[o] == shift[owner[at / kUnit]];
    }
    const uintptr_t dev = want ? kHost + at + shift[owner[at / kUnit]] : 0;
    if (reachable(kHost + at, bytes, write, ask) != dev) {
      std::printf("FAIL at %zu bytes %zu write %d\n", at, bytes, write);
      return 1;
    }
    ++n;
    yes += want;
    joined += want && owner[at / kUnit] != owner[(at + bytes - 8) / kUnit];
  }
  if (yes < 1000 || joined < 1000) {
    std::printf("FAIL %lld %lld\n", yes, joined);
    return 1;
  }
  std::printf("OK %lld\n", n);
  return 0;
}
