"""How the resident launches of a batch share the device: every combination of
cluster counts that the split chooses is resident at once, whatever the GPCs it
lands on (CPU, the rule compiled on its own)."""
import functools
import itertools
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1401_1112_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "split.h"
int main() {
  ats::SplitIn in;
  while (std::scanf("%d %d %d %d %d %d %d %d %d %d %lf %lf %lf %lf %lf %lf %lf %d", &in.slots, in.size, in.size + 1,
                    in.size + 2, in.fit, in.fit + 1, in.fit + 2, in.count, in.count + 1, in.count + 2, in.work,
                    in.work + 1, in.work + 2, in.work + 3, in.longest, in.longest + 1, in.longest + 2,
                    &in.singles) == 18) {
    int k[3];
    ats::split_clusters(in, k);
    std::printf("%d %d %d\n", k[0], k[1], k[2]);
  }
  return 0;
}
"""

# SMs per GPC that clusters of more than two CTAs can use, by the device's own counts of resident clusters of 1 .. 16
# CTAs: 16: 7, 12: 8, 10: 13, 9: 15, 8: 15, 6: 23, 5: 28, 4: 36, 3: 46
GPCS = {"gb300": (152, (20, 20, 20, 20, 20, 18, 18, 12)), "even": (144, (18,) * 8), "small": (40, (20, 14, 6))}


@functools.lru_cache(maxsize=None)
def _placed(free, todo):
    """Whether the clusters `todo` (descending) find room in whichever GPC each one before them took."""
    if not todo:
        return True
    at = {i: f for i, f in enumerate(free) if f >= todo[0]}
    return bool(at) and all(_placed(tuple(sorted(free[:i] + (f - todo[0],) + free[i + 1:])), todo[1:])
                            for i, f in at.items())


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("split")
    (d / "split.cpp").write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-I", CSRC, str(d / "split.cpp"), "-o", str(d / "split")], check=True)

    def run(cases):
        text = "\n".join(" ".join(str(v) for v in c) for c in cases)
        out = subprocess.run([str(d / "split")], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]

    return run


@pytest.mark.parametrize("gpcs", GPCS)
@pytest.mark.parametrize("sizes", [(16, 8, 4), (12, 8, 2), (8, 4, 2)])
def test_chosen_clusters_are_resident_at_once(split, gpcs, sizes):
    slots, cap = GPCS[gpcs]
    fit = [sum(c // s for c in cap) for s in sizes]
    rng = random.Random(1)
    cases = []
    for _ in range(400):
        count = [rng.choice([0, 1, 5, 200]) for _ in range(3)]
        work = [rng.uniform(1, 40) * (n > 0) for n in count] + [rng.choice([0.0, 1.0, 10.0])]
        longest = [min(w, rng.uniform(0.01, 0.3) * w) for w in work[:3]]
        cases.append([slots, *sizes, *fit, *count, *work, *longest, 100 if work[3] else 0])
    for c, k in zip(cases, split(cases)):
        count, singles = c[7:10], c[17]
        assert all((n > 0) == (m > 0) and m <= max(1, n) for n, m in zip(count, k)), (c, k)
        used = sum(n * s for n, s in zip(k, sizes))
        one_each = [int(n > 0) for n in count]
        if list(k) == one_each:
            continue  # also where nothing fits
        share = max(1, -(-slots * c[13] // sum(c[10:14]))) if singles else 0
        assert used + share <= slots, (c, k)
        todo = tuple(itertools.chain.from_iterable([s] * n for s, n in zip(sizes, k)))
        assert _placed(tuple(sorted(cap)), todo), (c, k)


def test_combination_that_waited_is_not_chosen(split):
    """512 levels of 64 .. 32 768 octs: 6 + 4 clusters of 16 and 8 would end
    first by their work alone, and cannot all be resident."""
    case = [152, 16, 8, 4, 7, 15, 36, 60, 80, 120, 96.0, 32.0, 16.0, 4.0, 2.0, 1.0, 0.5, 250]
    (k,) = split([case])
    assert k != (6, 4, 4) and 2 * k[0] + k[1] <= 15
