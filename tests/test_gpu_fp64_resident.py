"""GPU parity of the FP64 resident solver's groups against the oracle.

An FP64 level runs on one CTA (up to 128 octs), on a cluster of 4, 8 or 16
CTAs (runs of at most 128 octs each) or, above 2 048 octs, on the whole-GPU
form; the sizes here sit at those edges.  Both sides stop on the certified
rule ||b - A x|| <= 5e-11 ||x||, lambda_min >= 1 bounds each solution's error
by its residual, so they differ by at most 1e-10 relative.
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


def _check(ats, ctx, lv, st, **kw):
    f = dict(face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)
    xr, info = oracle.pcg(oracle.assemble(lv, st.dt, st.K, st.E, s=st.s, src=st.src, **f), st.E, tol=TOL,
                          stop_rule=oracle.STOP_CERTIFIED)
    assert info["status"] == 0
    L = ats.Level(ctx, lv)
    L.build(st.dt, st.K, st.E, s=st.s, src=st.src, **f)
    xs = []
    for _ in range(2):  # run to run
        x = st.E.copy()
        code, stats = L.solve(x, tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_FP64, **kw)
        assert code == 0, stats
        assert stats["err_bound"] <= TOL
        xs.append(x)
    L.close()
    np.testing.assert_array_equal(xs[0], xs[1])
    assert np.linalg.norm(xs[0] - xr) <= PAR * np.linalg.norm(xr)
    nl = ~lv.leaf_cells()
    np.testing.assert_array_equal(xs[0][nl], st.E[nl])


@pytest.mark.parametrize("dims", [(1, 1, 1), (8, 4, 4), (43, 3, 1), (57, 9, 1), (25, 41, 1), (16, 16, 8), (683, 3, 1),
                                  (19, 21, 23)],
                         ids=["1", "128", "129", "513", "1025", "2048", "2049", "9177"])
def test_group_edges_match_oracle(ats, ctx, dims):
    """1 .. 128 octs: one CTA; to 512, 1 024, 2 048: clusters; above: the whole GPU (with idle threads in each
    CTA's run and a last run that is shorter)."""
    rng = np.random.default_rng(sum(dims))
    dx = 1.0 / (2 * max(dims))
    lv = W.box_level(*dims, dx, [(W.DIRICHLET, 1.0), (W.NEUMANN, 0.0), (W.ROBIN, 0.3), (W.DIRICHLET, 1.0),
                                 (W.ROBIN, 0.8), None])
    N, nf = lv.n_cell, lv.n_face
    st = W.Step(dt=30 * dx * dx / 2, K=np.exp(rng.standard_normal(N)), E=rng.uniform(0.5, 1.5, N),
                face_K=np.exp(rng.standard_normal(nf)), face_E=rng.uniform(0.0, 2.0, nf),
                face_F=rng.uniform(-0.05, 0.05, nf))
    _check(ats, ctx, lv, st)


@pytest.mark.parametrize("form", ["cta", "cluster", "grid"])
@pytest.mark.parametrize("seed", [31, 32])
def test_irregular_levels_with_shift_match_oracle(ats, ctx, seed, form):
    """Random oct unions with non-leaf cells, every interface kind, a diagonal shift and a source on each group kind
    (the whole GPU: more CTAs than octs)."""
    lv, st = W.random_amr_level(seed, n_box=4, box_hi=8)
    rng = np.random.default_rng(seed)
    st.s, st.src = rng.uniform(0, 2, lv.n_cell), rng.uniform(-0.1, 0.1, lv.n_cell)
    kw = {"cta": dict(res_cta_octs=4096), "cluster": dict(res_cta_octs=-1, res_cluster=2),
          "grid": dict(sched=ats.ATS_SCHED_GRID, res_max_octs=8)}[form]
    _check(ats, ctx, lv, st, **kw)


def test_levels_in_lockstep_give_their_solo_bits(ats, ctx):
    """18 levels above the clusters' limit in one launch (16 in flight, the others as places free up), beside two small
    ones: each gives the bits it gives alone, and one is checked against the oracle."""
    rng = np.random.default_rng(5)
    cases = [W.random_box_solve(rng, o, robin=True) for o in np.linspace(2100, 6000, 18).tolist() + [60, 900]]
    levels, solo = [], []
    opts = dict(tol=TOL, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_FP64)
    for lv, st in cases:
        L = ats.Level(ctx, lv)
        L.build(st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F)
        x = st.E.copy()
        code, stats = L.solve(x, **opts)
        assert code >= 0, stats
        levels.append(L)
        solo.append((x, stats))
    B = ats.Batch(ctx, levels, **opts)
    xs = [st.E.copy() for _, st in cases]
    code, stats = B.solve(xs)
    assert code >= 0
    for (x, s), y, t in zip(solo, xs, stats):
        np.testing.assert_array_equal(y, x)
        assert s == t
    lv, st = cases[3]
    xr, _ = oracle.pcg(oracle.assemble(lv, st.dt, st.K, st.E, face_K=st.face_K, face_E=st.face_E, face_F=st.face_F),
                       st.E, tol=TOL, stop_rule=oracle.STOP_CERTIFIED)
    assert np.linalg.norm(xs[3] - xr) <= PAR * np.linalg.norm(xr)
    B.close()
    for L in levels:
        L.close()
