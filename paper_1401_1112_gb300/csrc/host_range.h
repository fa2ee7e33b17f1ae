// Which host results the device writes itself.
#pragma once

#include <cstddef>
#include <cstdint>

namespace ats {

// Host memory [lo, hi) that the device can write, and the device's address of lo.
struct HostRange {
  uintptr_t lo = 0, hi = 0, dev = 0;
};

// For each of n host arrays (len[k] doubles at x[k]): dev[k] = the device's
// address of x[k] where the whole array is pinned, else null.  query(p) gives
// the pinned range around p, empty where there is none.  Asked at every run: an
// address says nothing about whether its memory is still pinned (unregistered,
// or freed and allocated again, between two runs).  Arrays that follow one
// another in one allocation cost one query.
template <typename Query>
void host_targets(double *const *x, const size_t *len, int n, double **dev, const Query &query) {
  HostRange r;
  for (int k = 0; k < n; ++k) {
    const uintptr_t a = (uintptr_t)x[k], b = a + len[k] * sizeof(double);
    if (a < r.lo || b > r.hi) r = query(x[k]);
    dev[k] = a >= r.lo && b <= r.hi ? (double *)(r.dev + (a - r.lo)) : nullptr;
  }
}

}  // namespace ats
