"""Which host results the device writes itself: pinned arrays, asked for anew at
every run.  The rule runs here on the CPU against a stand-in for the driver's
pointer query; the solves need a GPU."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import workloads as W

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1401_1112_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "host_range.h"

static bool pinned = false;
static double a[64];

static bool query(double *p, void **d) {
  *d = (char *)p + 4096;  // the device's view lies elsewhere
  return pinned;
}
static void check(bool ok, const char *what) {
  if (!ok) {
    std::printf("%s\n", what);
    std::exit(1);
  }
}
int main() {
  double *x[2] = {a, a + 32}, *dev[2];
  for (int run = 0; run < 4; ++run) {  // the same addresses, pinned in every second run
    pinned = run & 1;
    ats::host_targets(x, 2, dev, query);
    for (int k = 0; k < 2; ++k)
      check(dev[k] == (pinned ? (double *)((char *)x[k] + 4096) : nullptr), "stale answer");
  }
  return 0;
}
"""


def test_pinned_state_is_asked_at_every_run(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "targets.cpp", tmp_path / "targets"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


@pytest.mark.gpu
def test_registering_an_array_between_runs_keeps_its_results():
    """A batch on the same numpy arrays, pageable, registered and unregistered
    in turn: the same bits each time."""
    import torch

    from paper_1401_1112_gb300 import ats, build

    build.build()
    rt = torch.cuda.cudart()
    rng = np.random.default_rng(8)
    cases = [W.random_box_solve(rng, o) for o in (70, 1300)]
    with ats.Context(0) as ctx:
        levels = []
        for lv, st in cases:
            L = ats.Level(ctx, lv)
            L.build(st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)
            levels.append(L)
        B = ats.Batch(ctx, levels, tol=5e-11, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_MIXED)
        xs, first = [st.E.copy() for _, st in cases], None
        for run in range(4):
            for x, (_, st) in zip(xs, cases):
                x[:] = st.E
                if run & 1:
                    assert int(rt.cudaHostRegister(x.ctypes.data, x.nbytes, 0)) == 0
            assert B.solve(xs)[0] == 0
            if run & 1:
                for x in xs:
                    assert int(rt.cudaHostUnregister(x.ctypes.data)) == 0
            if first is None:
                first = [x.copy() for x in xs]
            for x, y in zip(xs, first):
                np.testing.assert_array_equal(x, y)
        B.close()
        for L in levels:
            L.close()
