"""Which group a mixed-precision level takes on the resident solver: by its octs
and the options' values, at the edges of the rule.

A batch of one level launches one group, so its launch shows the group: [CTAs
of the larger clusters, of the base clusters, single CTAs beside them]; a level
for one CTA is offered every CTA of the device.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


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


def _run(ats, ctx, dims, **kw):
    rng = np.random.default_rng(sum(dims))
    lv = W.box_level(*dims, 1.0 / (2 * max(dims)), [(W.DIRICHLET, 1.0), None, None, (W.ROBIN, 0.4), None, None])
    K, E = np.exp(rng.standard_normal(lv.n_cell)), rng.uniform(0.5, 1.5, lv.n_cell)
    L = ats.Level(ctx, lv)
    L.build(5 * lv.dx ** 2, K, E, face_E=rng.uniform(0, 2, lv.n_face))
    B = ats.Batch(ctx, [L], tol=5e-11, stop_rule=ats.ATS_STOP_CERTIFIED, precision=ats.ATS_PREC_MIXED, **kw)
    x = E.copy()
    code, stats = B.solve([x])
    assert code == 0, stats
    grids = B.kernel_stats()["res_grids"]
    B.close()
    L.close()
    big, base = int(grids[0]), int(grids[1])
    return x, (big or (base if base <= 16 else 1))


@pytest.mark.parametrize("dims,limit,group", [((16, 16, 8), 0, 1), ((683, 3, 1), 0, 4), ((24, 16, 16), 0, 4),
                                              ((1229, 5, 1), 0, 8), ((32, 24, 16), 0, 8), ((12289, 1, 1), 0, 16),
                                              ((16, 16, 8), 32768, 1), ((32, 16, 16), 32768, 4),
                                              ((2731, 3, 1), 32768, 8), ((32, 32, 16), 32768, 8),
                                              ((113, 29, 5), 32768, 16)],
                         ids=["2048", "2049", "6144", "6145", "12288", "12289", "2048-long", "8192-long", "8193-long",
                              "16384-long", "16385-long"])
def test_group_by_size(ats, ctx, dims, limit, group):
    x, g = _run(ats, ctx, dims, res_max_octs=limit)
    assert g == group
    if limit == 0:  # the default's value written out: the same group and bits
        y, h = _run(ats, ctx, dims, res_max_octs=16384)
        assert h == group
        np.testing.assert_array_equal(x, y)
        y, h = _run(ats, ctx, dims, res_cta_octs=2048)
        assert h == group
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("dims,kw", [((16, 16, 8), dict(res_cta_octs=-1)), ((24, 16, 16), {}), ((16, 16, 16), {}),
                                     ((32, 16, 16), dict(res_max_octs=32768)), ((1229, 5, 1), {}),
                                     ((32, 32, 16), dict(res_max_octs=32768))],
                         ids=["512-x4", "1536-x4", "1024-x4", "2048-x4", "769-x8", "2048-x8"])
def test_same_bits_with_the_state_in_global_memory(ats, ctx, dims, kw):
    """Both register layouts on the clusters of the rule."""
    x, g = _run(ats, ctx, dims, **kw)
    y, h = _run(ats, ctx, dims, res_state=1, **kw)
    assert g == h
    np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("prec,limit,shapes", [("mixed", 0, 8), ("mixed", 1024, 8), ("mixed", 512, 9), ("fp64", 0, 9),
                                               ("fp64", 2048, 8)])
def test_autotuner_leaves_out_the_batchs_own_shape_alone(ats, ctx, prec, limit, shapes):
    """Eight resident shapes and the batch's own: the one that is its own, by
    the default limit or the given one, is not timed twice, and no other is
    left out (FP64 by default: 256 threads, 4 CTAs, 128 octs on one CTA)."""
    rng = np.random.default_rng(1)
    levels = []
    for o in (90, 1500):
        lv, st = W.random_box_solve(rng, o, dt_hi=1.0)
        L = ats.Level(ctx, lv)
        L.build(st.dt, st.K, st.E, face_E=st.face_E, face_F=st.face_F)
        levels.append((L, st))
    precision = ats.ATS_PREC_MIXED if prec == "mixed" else ats.ATS_PREC_FP64
    B = ats.Batch(ctx, [L for L, _ in levels], tol=5e-11, stop_rule=ats.ATS_STOP_CERTIFIED, precision=precision,
                  res_cta_octs=limit)
    r = B.autotune([st.E.copy() for _, st in levels], reps=1)
    assert r["candidates"] == shapes
    B.close()
    for L, _ in levels:
        L.close()
