"""Which host results the device writes itself: arrays that are pinned from end
to end, asked for anew at every run.  The rule runs here on the CPU against a stand-in for the driver's
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

static double a[64];
static uintptr_t lo, hi;  // what is pinned
static int asked;

static ats::HostRange query(const void *p) {
  ++asked;
  const uintptr_t at = (uintptr_t)p;
  ats::HostRange r;
  if (at >= lo && at < hi) r = {lo, hi, lo + 4096};  // the device's view lies elsewhere
  return r;
}
static void pin(int first, int last) {
  lo = (uintptr_t)(a + first);
  hi = (uintptr_t)(a + last);
}
static void check(bool ok, const char *what) {
  if (!ok) {
    std::printf("%s\n", what);
    std::exit(1);
  }
}
static double *at_dev(double *p) { return (double *)((char *)p + 4096); }
int main() {
  double *x[2] = {a, a + 32}, *dev[2];
  const size_t len[2] = {32, 32};
  for (int run = 0; run < 4; ++run) {  // the same addresses, pinned in every second run
    pin(0, run & 1 ? 64 : 0);
    ats::host_targets(x, len, 2, dev, query);
    for (int k = 0; k < 2; ++k) check(dev[k] == (run & 1 ? at_dev(x[k]) : nullptr), "stale answer");
  }
  for (int last = 1; last <= 64; ++last) {  // pinned up to somewhere inside an array
    pin(0, last);
    ats::host_targets(x, len, 2, dev, query);
    for (int k = 0; k < 2; ++k) check(dev[k] == (last >= 32 * (k + 1) ? at_dev(x[k]) : nullptr), "partly pinned");
  }
  pin(8, 64);  // ... and from somewhere inside one
  ats::host_targets(x, len, 2, dev, query);
  check(!dev[0] && dev[1] == at_dev(x[1]), "pinned from the middle");
  pin(0, 64);
  asked = 0;
  ats::host_targets(x, len, 2, dev, query);
  check(asked == 1, "one query for one allocation");
  return 0;
}
"""


def test_only_wholly_pinned_arrays_and_asked_at_every_run(tmp_path):
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


@pytest.mark.gpu
@pytest.mark.parametrize("first,last,status", [(0.0, 1.0, 0), (0.0, 0.5, -7), (0.25, 1.0, 0), (0.3, 0.6, 0)])
def test_partly_registered_array_is_not_written_by_the_device(first, last, status):
    """A slab of two levels' arrays, the start guess taken from E^n on the
    device.  An array registered from end to end is written by the device, one
    registered in part is copied: CUDA takes a copy that begins in pageable
    memory, and refuses one that begins registered and ends beyond it (the
    solve then ends with ATS_ERR_CUDA).  Every run that is taken has the
    pageable slab's bits."""
    import torch

    from paper_1401_1112_gb300 import ats, build

    build.build()
    rt = torch.cuda.cudart()
    rng = np.random.default_rng(9)
    cases = [W.random_box_solve(rng, o) for o in (600, 1300)]
    off = np.cumsum([0] + [lv.n_cell for lv, _ in cases])
    slab = np.empty(off[-1])
    with ats.Context(0) as ctx:
        levels, out = [], []
        for lv, st in cases:
            L = ats.Level(ctx, lv)
            L.build(st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)
            levels.append(L)
        B = ats.Batch(ctx, levels, tol=5e-11, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_MIXED,
                      x0=ats.ATS_X0_E_OLD)
        i, j = int(first * off[-1]), int(last * off[-1])
        for part in (False, True, False):
            slab[:] = 0.0
            if part:
                assert int(rt.cudaHostRegister(slab[i:].ctypes.data, 8 * (j - i), 0)) == 0
            code = B.solve([slab[off[k]:off[k + 1]] for k in range(2)])[0]
            if part:
                assert int(rt.cudaHostUnregister(slab[i:].ctypes.data)) == 0
            assert code == (status if part else 0)
            if code == 0:
                out.append(slab.copy())
        for x in out[1:]:
            np.testing.assert_array_equal(x, out[0])
        B.close()
        for L in levels:
            L.close()
