// hostbuf.h -- which host buffers of the caller a kernel may read or write itself, and how
// long.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace dfn {

// What the driver says of a host address: the device's address of it, and the device range
// of the allocation or registration that holds it.
struct HostPart {
  bool pinned;    // page-locked host memory
  bool writable;  // not registered read-only
  uintptr_t dev, start;
  size_t size;
};

// The device's address of the `bytes` from `host` on if a kernel may touch them all, else 0.
// `ask` gives the HostPart of an address.  Where one allocation or registration ends before
// the buffer does, the next has to begin right there, on the device too: both ends alone say
// nothing about what lies between them (memory that the device cannot reach has no device
// address, yet the ends may lie as far apart on the device as on the host).
template <class Ask>
uintptr_t reachable(uintptr_t host, size_t bytes, bool write, Ask ask) {
  uintptr_t dev = 0;
  for (size_t done = 0; done < bytes;) {
    const HostPart p = ask(host + done);
    if (!p.pinned || !p.dev || (write && !p.writable)) return 0;
    if (p.dev < p.start || p.dev - p.start >= p.size) return 0;
    if (done == 0) dev = p.dev;
    if (p.dev != dev + done) return 0;
    const size_t rest = p.size - (p.dev - p.start);
    done = rest < bytes - done ? done + rest : bytes;
  }
  return dev;
}

// Starts n transfers to or from the caller's buffer, up to the first that fails (issue(k)
// gives a non-zero code), and then waits for those started in either case: when this returns
// the device is done with the buffer.  The first code is returned; wait(failed) gives the
// wait's own.
template <class Issue, class Wait>
int transfer_all(int n, Issue issue, Wait wait) {
  int rc = 0;
  for (int k = 0; k < n && !rc; ++k) rc = issue(k);
  const int waited = wait(rc != 0);
  return rc ? rc : waited;
}

}  // namespace dfn
