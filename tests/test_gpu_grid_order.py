"""Mixed-precision levels on the whole-GPU form whose octs are in no order, whose
energies leave the fixed-point sum's range, or that run beside a larger level.

Both sides stop on ||b - A x|| <= 5e-11 ||x||, lambda_min >= 1 bounds each
solution's error by its residual: they differ by at most 1e-10 relative.  The
same solve twice, and alone or in a batch, gives the same bits.
"""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

TOL, PAR = 5e-11, 1e-10


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


def _box(rng, dims, cfl, shuffled=False):
    dx = 1.0 / (2 * max(dims))
    lv = W.box_level(*dims, dx, [(W.DIRICHLET, 1.0), (W.NEUMANN, 0.0), None, (W.ROBIN, 0.3), None, None])
    if shuffled:
        to = rng.permutation(lv.n_oct)  # oct o becomes oct to[o]
        xyz = np.empty_like(lv.oct_xyz)
        xyz[to] = lv.oct_xyz
        cell = 8 * to[lv.face_cell // 8] + lv.face_cell % 8
        order = np.lexsort((lv.face_dir, cell))
        lv = W.LevelDesc(xyz, None, dx, cell[order].astype(np.int32), lv.face_dir[order], lv.face_kind[order],
                         lv.face_rel[order], lv.face_alpha[order])
    nf = lv.n_face
    return lv, W.Step(dt=cfl * dx * dx / 2, K=np.exp(0.5 * rng.standard_normal(lv.n_cell)),
                      E=rng.uniform(0.0, 2.0, lv.n_cell), face_K=np.ones(nf), face_E=rng.uniform(0.0, 2.0, nf),
                      face_F=rng.uniform(-0.05, 0.05, nf))


def _level(ats, ctx, lv, st, scale=1.0):
    L = ats.Level(ctx, lv)
    L.build(st.dt, st.K, scale * st.E, face_K=st.face_K, face_E=scale * st.face_E, face_F=scale * st.face_F)
    return L


def _opts(ats, **kw):
    return dict(tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_MIXED, **kw)


def _system(lv, st):
    return oracle.assemble(lv, st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)


def _oracle_x(lv, st):
    x, info = oracle.pcg(_system(lv, st), st.E, tol=TOL, stop_rule=oracle.STOP_CERTIFIED)
    assert info["status"] == 0
    return x


@pytest.mark.parametrize("dims", [(26, 26, 26), (43, 42, 42)], ids=["run-116", "run-500"])
def test_octs_in_no_order(ats, ctx, dims):
    """Random order: nearly every face of a run of 116 octs, and of one of 500
    (about 3 000 faces, twice what a CTA stages), lies in another CTA's run.
    Which faces are staged follows the order of atomics, the bits do not."""
    lv, st = _box(np.random.default_rng(dims[0]), dims, 3.0, shuffled=True)
    L = _level(ats, ctx, lv, st)
    xs, all_stats = [], []
    for _ in range(3):
        x = st.E.copy()
        code, stats = L.solve(x, **_opts(ats))
        assert code == 0, stats
        xs.append(x)
        all_stats.append(stats)
    L.close()
    for x, s in zip(xs[1:], all_stats[1:]):
        np.testing.assert_array_equal(x, xs[0])
        assert s == all_stats[0]
    ref = _oracle_x(lv, st)
    assert np.linalg.norm(xs[0] - ref) <= PAR * np.linalg.norm(ref)


def test_energies_beyond_the_fixed_point_range(ats, ctx):
    """All energies times a power of two that takes the first r.z past 1e37,
    where the p.q sum goes its slow way; later steps, with a smaller r.z, take
    the fixed-point words.  The solution scales with the energies."""
    lv, st = _box(np.random.default_rng(3), (12, 11, 10), 1.0)
    S = _system(lv, st)
    r, _ = S.residual(st.E)
    rz = float((r * r / S.diag).sum())
    scale = 2.0 ** np.floor(np.log2(np.sqrt(4.8e37 / rz)))
    assert scale ** 2 * rz > 1.1e37 and scale ** 2 * max((r * r).sum(), (st.E ** 2).sum()) < 3e38
    opts = _opts(ats, sched=ats.ATS_SCHED_GRID, res_max_octs=8)
    L = _level(ats, ctx, lv, st, scale)
    xs = []
    for _ in range(2):
        x = scale * st.E
        code, stats = L.solve(x, **opts)
        assert code == 0, stats
        xs.append(x)
    L.close()
    np.testing.assert_array_equal(xs[0], xs[1])
    ref = _oracle_x(lv, st)
    assert np.linalg.norm(xs[0] / scale - ref) <= PAR * np.linalg.norm(ref)


def test_same_bits_beside_a_larger_level(ats, ctx):
    """Levels of both on-chip layouts (runs of 116 and 1 115 octs) alone, and in
    a batch whose largest level streams part of its octs."""
    rng = np.random.default_rng(12)
    cases = [_box(rng, dims, 3.0) for dims in ((26, 26, 26), (55, 55, 56), (75, 70, 64))]
    levels = [_level(ats, ctx, lv, st) for lv, st in cases]
    solo = []
    for L, (_, st) in zip(levels[:2], cases):
        x = st.E.copy()
        code, stats = L.solve(x, **_opts(ats))
        assert code == 0, stats
        solo.append((x, stats))
    B = ats.Batch(ctx, levels, **_opts(ats))
    xs = [st.E.copy() for _, st in cases]
    code, stats = B.solve(xs)
    assert code == 0, stats
    for (x, s), y, t in zip(solo, xs, stats):
        np.testing.assert_array_equal(y, x)
        assert s == t
    B.close()
    for L in levels:
        L.close()
