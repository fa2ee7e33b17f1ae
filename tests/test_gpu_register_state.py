"""The mixed-precision resident solver with its CG state in registers against
the same solve with every array in global memory: bitwise the same results.

Where a value lives does not change what is computed, so the tolerance is
zero.  Sizes: the edges of the two register layouts (1 024 and 2 048 octs per
CTA), a run that ends inside a warp, clusters, and levels with non-leaf cells.
The whole-GPU form has no global-memory counterpart: its longer runs are
compared with the tick path, both certified to 5e-11, within 1e-10.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

TOL = 5e-11


@pytest.fixture(scope="module")
def ats():
    from paper_1401_1112_gb300 import ats as A
    from paper_1401_1112_gb300 import build

    build.build()
    return A


@pytest.fixture(scope="module")
def ctx(ats):
    c = ats.Context(0)
    yield c
    c.close()


def _box(dims):
    rng = np.random.default_rng(sum(dims))
    dx = 1.0 / (2 * max(dims))
    lv = W.box_level(*dims, dx, [(W.DIRICHLET, 1.0), (W.NEUMANN, 0.0), (W.ROBIN, 0.3), (W.DIRICHLET, 1.0),
                                 (W.ROBIN, 0.8), None])
    N, nf = lv.n_cell, lv.n_face
    return lv, W.Step(dt=30 * dx * dx / 2, K=np.exp(rng.standard_normal(N)), E=rng.uniform(0.5, 1.5, N),
                      face_K=np.exp(rng.standard_normal(nf)), face_E=rng.uniform(0.0, 2.0, nf),
                      face_F=rng.uniform(-0.05, 0.05, nf))


def _solve(ats, ctx, lv, st, **kw):
    L = ats.Level(ctx, lv)
    L.build(st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)
    x = st.E.copy()
    code, stats = L.solve(x, tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_MIXED, **kw)
    L.close()
    assert code == 0, stats
    assert stats["err_bound"] <= TOL
    return x, stats


@pytest.mark.parametrize("dims,kw", [((1, 1, 1), {}), ((16, 8, 8), {}), ((41, 25, 1), dict(res_cta_octs=2048)),
                                     ((16, 16, 8), dict(res_cta_octs=2048)), ((41, 25, 1), {}), ((16, 16, 16), {}),
                                     ((27, 19, 8), dict(res_max_octs=16384)), ((27, 19, 8), {}),
                                     ((16, 16, 16), dict(res_max_octs=16384, res_cluster=2)),
                                     ((9, 9, 9), dict(res_cta_octs=-1, res_cluster=3))],
                         ids=["1", "1024-cta", "1025-cta", "2048-cta", "257-x4", "1024-x4", "1026-x4", "513-x8",
                              "2048-x2", "243-x3"])
def test_same_bits_as_global_state(ats, ctx, dims, kw):
    lv, st = _box(dims)
    x, stats = _solve(ats, ctx, lv, st, **kw)
    xg, sg = _solve(ats, ctx, lv, st, res_state=1, **kw)
    np.testing.assert_array_equal(x, xg)
    assert stats == sg


@pytest.mark.parametrize("kw", [dict(res_cta_octs=4096), dict(res_cta_octs=-1, res_cluster=4)], ids=["cta", "x4"])
@pytest.mark.parametrize("seed", [41, 42])
def test_same_bits_with_non_leaf_cells(ats, ctx, seed, kw):
    lv, st = W.random_amr_level(seed, n_box=4, box_hi=8)
    x, stats = _solve(ats, ctx, lv, st, **kw)
    xg, sg = _solve(ats, ctx, lv, st, res_state=1, **kw)
    np.testing.assert_array_equal(x, xg)
    assert stats == sg


@pytest.mark.parametrize("dims", [(54, 54, 53), (58, 58, 50), (68, 68, 67), (68, 68, 68)],
                         ids=["run-1017", "run-1107", "run-2039", "run-2069"])
def test_whole_gpu_layout_edge(ats, ctx, dims):
    """154 548 and 168 200 octs over 152 CTAs: the two register layouts; 309 808 and 314 432: just within and just
    beyond what a CTA keeps on chip."""
    lv, st = _box(dims)
    x, _ = _solve(ats, ctx, lv, st, sched=ats.ATS_SCHED_GRID)
    xt, _ = _solve(ats, ctx, lv, st, sched=ats.ATS_SCHED_TICK)
    assert np.linalg.norm(x - xt) <= 1e-10 * np.linalg.norm(xt)


def test_whole_gpu_tail_with_non_leaf_cells(ats, ctx):
    """A level beyond the on-chip capacity whose every 1 000th oct has refined cells: the octs in global memory keep
    them out of the stencil as the others do."""
    lv, st = _box((80, 70, 60))
    leaf = np.full(lv.n_oct, 0xFF, np.uint8)
    inner = np.all((lv.oct_xyz > 0) & (lv.oct_xyz < np.array([79, 69, 59])), axis=1)
    leaf[np.nonzero(inner)[0][::1000]] = 0x5A
    lv.leaf = leaf
    x, _ = _solve(ats, ctx, lv, st)
    xt, _ = _solve(ats, ctx, lv, st, sched=ats.ATS_SCHED_TICK)
    assert np.linalg.norm(x - xt) <= 1e-10 * np.linalg.norm(xt)
    nl = ~lv.leaf_cells()
    np.testing.assert_array_equal(x[nl], st.E[nl])
