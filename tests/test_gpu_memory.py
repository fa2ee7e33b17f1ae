"""What a whole-GPU plan allocates counts: against the context's budget and in
the bytes it reports."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,dims", [("fp64", (16, 16, 9)), ("mixed", (32, 32, 17))], ids=["fp64", "mixed"])
def test_whole_gpu_plan_counts_against_the_budget(prec, dims):
    """The words of the grid barrier (5 x 64 ints) and of the partial sums (2
    sets x 3 sums per CTA, one CTA per SM, and a spare row each) are what such
    a plan holds beside a tick-path plan of the same level; a budget one byte
    below it refuses the solve, the exact one takes it."""
    import torch

    from paper_1401_1112_gb300 import ats, build

    build.build()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lv = W.box_level(*dims, 1.0 / (2 * max(dims)))
    precision = ats.ATS_PREC_FP64 if prec == "fp64" else ats.ATS_PREC_MIXED

    E = np.linspace(0.5, 1.5, lv.n_cell)

    def used(sched, budget=0):
        with ats.Context(0, mem_budget_bytes=budget) as ctx:
            L = ats.Level(ctx, lv)
            L.build(1e-3, np.ones(lv.n_cell), E)
            x = E.copy()
            code, _ = L.solve(x, precision=precision, sched=sched)
            bytes_used = ctx.memory()[0]
            L.close()
            return code, bytes_used

    code, tick = used(ats.ATS_SCHED_TICK)
    assert code == 0
    code, grid = used(ats.ATS_SCHED_AUTO)
    assert code == 0
    assert grid - tick >= 5 * 64 * 4 + 2 * 3 * 8 * (sms + 1)
    assert used(ats.ATS_SCHED_AUTO, grid)[0] == 0
    assert used(ats.ATS_SCHED_AUTO, grid - 1)[0] == ats.ATS_ERR_OVER_BUDGET
