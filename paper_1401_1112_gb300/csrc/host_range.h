// Which host results the device writes itself.
#pragma once

#include <cstddef>
#include <cstdint>

namespace ats {

// For each of n host arrays x[k]: dev[k] = the device's address of x[k] where
// the memory is pinned, else null.  query(p, &d) says whether p lies in memory
// the device can write, and at which device address.  Asked at every run: an
// address says nothing about whether its memory is still pinned (unregistered,
// or freed and allocated again, between two runs).
template <typename Query>
void host_targets(double *const *x, int n, double **dev, const Query &query) {
  for (int k = 0; k < n; ++k) {
    void *d = nullptr;
    dev[k] = query(x[k], &d) ? (double *)d : nullptr;
  }
}

}  // namespace ats
