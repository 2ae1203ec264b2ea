"""Multipath-lifetime plan of the FP64 form where a change lies at the threshold: the plan is taken from FP32 synthesis records,
and a share within their rounding of the threshold has to be decided by the FP64 outputs."""
import os

import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


@pytest.mark.parametrize("offset", [-1e-9, 1e-9, -1e-4, 1e-4])
def test_share_at_the_threshold(offset):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    paths = I.PathSet.from_npz(os.path.join(GOLD, "pathset_canyon_seed0.npz"))
    tg, fg = I.TimeGrid(0.0, 2e-3, 400), I.FreqGrid(60e9, 1e9, 8)
    with drt.Context(0) as ctx:
        link = ctx.load(I.scene_canyon(0), paths)
        r = {k: v.cpu().numpy() for k, v in link.extrapolate(tg, fg, drt.FP64).items() if v is not None}
        valid = r["flags"] == 0
        pw = np.where(valid, (r["amp"] ** 2).sum(-1), 0.0)
        tot = pw.sum(1)
        on = valid[1:] != valid[:-1]
        share = np.where(valid[1:], pw[1:] / tot[1:, None], pw[:-1] / tot[:-1, None])[on]
        for x in np.sort(share)[[-1, -5, -40]]:
            s = float(x) * (1 + offset)   # FP64 sums agree to ~1e-15, far inside the offset
            want = np.zeros(tg.n_steps, bool)
            want[1:] = (on & np.where(valid[1:], pw[1:] >= s * tot[1:, None], pw[:-1] >= s * tot[:-1, None])).any(1)
            _, major = link.lifetime_windows(tg, fg, s, 1, 50, drt.FP64)
            assert np.array_equal(major, want)
