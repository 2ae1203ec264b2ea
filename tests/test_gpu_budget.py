"""Calls at the smallest HBM budget: a route that needs more scratch gives way to the one that needs less."""
import os

import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


@pytest.mark.parametrize("extra", [0, 1 << 18, 1 << 20, 1 << 22])
def test_lifetime_plan_at_the_smallest_budget(extra):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    scene, paths = I.scene_canyon(0), I.PathSet.from_npz(os.path.join(GOLD, "pathset_canyon_seed0.npz"))
    tg, fg = I.TimeGrid(0.0, 2e-3, 400), I.FreqGrid(60e9, 1e9, 8)

    def plan(budget, share):
        with drt.Context(0, hbm_budget=budget) as ctx:
            try:
                return ctx.load(scene, paths).lifetime_windows(tg, fg, share, 1, 50, drt.FP64)[1]
            except drt.DrtError as e:
                assert e.code == drt.DRT_ENOMEM
                return None

    lo, hi = 1 << 16, 1 << 30   # a share of 0 takes the FP64 outputs: the least that any call needs
    while hi - lo > 1 << 16:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if plan(mid, 0.0) is not None else (mid, hi)
    got = plan(hi + extra, 0.01)
    assert got is not None and np.array_equal(got, plan(0, 0.01))
