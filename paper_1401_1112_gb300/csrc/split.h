// How the resident launches of a batch share the device.
#pragma once

#include <algorithm>
#include <cmath>

namespace ats {

// Three cluster classes, largest clusters first (count 0: none of that class),
// and the single CTAs.
struct SplitIn {
  int slots;          // CTAs resident at once
  int size[3];        // CTAs per cluster
  int fit[3];         // clusters of that size alone that are resident at once
  int count[3];       // solves
  double work[4];     // SM-time of each class's solves, the single CTAs' last
  double longest[3];  // ... of its longest solve
  int singles;        // solves on single CTAs
};

// Whether k[] clusters of the three classes are resident together.  A cluster
// takes its SMs from one GPC, so the total alone does not tell: a cluster of t
// CTAs leaves room for ceil(t / s) fewer clusters of s.  Measured on a GB300,
// whose GPCs give clusters 20 (five of them), 18 (two) and 12 SMs -- 7 clusters
// of 16, 15 of 8 or 36 of 4 CTAs: 6 + 4 or 5 + 6 clusters of 16 and 8, 128 of
// the 152 SMs and one of 8 too many, leave the smaller ones waiting for the end
// of a launch, 512 levels in 23.6 ms; 6 + 3 run in 13.4.
inline bool split_fits(const SplitIn &in, const int (&k)[3]) {
  for (int q = 0; q < 3; ++q) {
    if (k[q] == 0) continue;
    int room = in.fit[q];
    for (int t = 0; t < q; ++t) room -= k[t] * ((in.size[t] + in.size[q] - 1) / in.size[q]);
    if (k[q] > room) return false;
  }
  return true;
}

// The counts of clusters that make the class that ends last end earliest (each
// class ends after its work over its slots, and not before its longest solve),
// out of every combination that is resident at once and leaves the single CTAs
// their share, so that the largest of them start at once; every slot left over
// runs single CTAs too, and a cluster that has emptied its queue goes on with
// them.  Where not even one cluster of each class fits, one of each: they run
// after one another.
inline void split_clusters(const SplitIn &in, int (&k)[3]) {
  const double sum = std::max(1e-300, in.work[0] + in.work[1] + in.work[2] + in.work[3]);
  const int c_min = in.singles > 0 ? std::max(1, (int)std::ceil(in.slots * in.work[3] / sum)) : 0;
  int lo[3], hi[3];
  for (int q = 0; q < 3; ++q) {
    lo[q] = in.count[q] > 0 ? 1 : 0;
    hi[q] = in.count[q] > 0 ? std::max(1, std::min(in.fit[q], in.count[q])) : 0;
    k[q] = lo[q];
  }
  const auto end_of = [&](int q, int n) {
    return in.count[q] > 0 ? std::max(in.work[q] / ((double)n * in.size[q]), in.longest[q] / in.size[q]) : 0.0;
  };
  double best = HUGE_VAL;
  int best_used = 0;
  for (int i = lo[0]; i <= hi[0]; ++i)
    for (int j = lo[1]; j <= hi[1]; ++j)
      for (int l = lo[2]; l <= hi[2]; ++l) {
        const int n[3] = {i, j, l};
        const int used = i * in.size[0] + j * in.size[1] + l * in.size[2];
        if (used + c_min > in.slots || !split_fits(in, n)) break;
        const double t = std::max(end_of(0, i), std::max(end_of(1, j), end_of(2, l)));
        if (t < best || (t == best && used < best_used)) {
          best = t;
          best_used = used;
          for (int q = 0; q < 3; ++q) k[q] = n[q];
        }
      }
}

}  // namespace ats
