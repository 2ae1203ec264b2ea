"""Steps that the FP32-bulk form hands to its redo: plates whose rims lie 2e-5 m beyond their reflection points, inside the bound on the
FP32 error, so that every path-step is redone (the batch's count says so) and its outputs can be held to the redo's own precision.
"""
import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TX, RX = np.array([0.0, 0.0, 5.0]), np.array([60.0, 3.0, 1.5])
VT, VR = np.array([3.0, -7.0, 0.5]), np.array([-20.0, 9.0, 0.0])


def plates(n, seed):
    """n plates at random places and slopes, each with both terminals in front of it."""
    rng = np.random.default_rng(seed)
    b = I._Builder("plates")
    mat = b.material(5.3, 0.1)
    body = b.body(np.array([30.0, 0.0, 0.0]), [4.0, 6.0, -2.0], [0, 0, 0])
    for _ in range(n):
        while True:
            q = rng.uniform([-20, -60, -40], [80, 60, 40])
            u1, u2 = TX - q, RX - q
            n1 = u1 / np.linalg.norm(u1) + u2 / np.linalg.norm(u2)
            n1 /= np.linalg.norm(n1)
            if min(u1 @ n1, u2 @ n1) > 5.0:
                break
        u = np.cross(n1, rng.normal(size=3))
        u /= np.linalg.norm(u)
        b.face(body, mat, q - (8.0 - 2e-5) * u, n1, u, 8.0, 9.0)
    return b.build((list(TX), list(VT), [0, 0, 0]), (list(RX), list(VR), [0, 0, 0]))


@pytest.fixture(scope="module")
def redone():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    n = 300
    scene, paths = plates(n, 1), I.chains_to_pathset([[(I.T_R, i)] for i in range(n)])
    tg, fg = I.TimeGrid(0.0, 1e-8, 8), I.FreqGrid(28e9, 400e6, 4)   # microns of motion
    with drt.Context(0) as ctx:
        link = ctx.load(scene, paths)
        H = torch.empty(tg.n_steps, fg.n_bins, dtype=torch.complex64, device="cuda")
        with ctx.batch([link], [tg], [fg], [H]) as b:
            b.run()
            assert b.info(redo=True)["redo_steps"] == n * tg.n_steps
        out = [{k: v.cpu().numpy() for k, v in link.extrapolate(tg, fg, p).items() if v is not None}
               for p in (drt.FP64, drt.FP32_BULK)]
    assert not out[0]["flags"].any() and not out[1]["flags"].any()
    return out


def test_delay_and_doppler(redone):
    """Delay in two-float numbers (2^-46 an operation, some ten of them); Doppler shift to its FP32 rounding (2^-24) and as much again."""
    a, b = redone
    assert (np.abs(b["tau"] / a["tau"] - 1) <= 2.0 ** -42).all()
    assert (np.abs(b["doppler"] - a["doppler"]) <= 2.0 ** -23 * np.abs(a["doppler"])).all()


def test_angles(redone):
    """Both forms round an angle to FP32: to the same or to neighbouring numbers."""
    a, b = redone
    assert (np.abs(b["angles"].astype(np.float64) - a["angles"]) <= np.spacing(np.abs(a["angles"]))).all()


@pytest.mark.parametrize("bins,bandwidth", [(4096, 3.7e8), (4096, 1.3e9), (4096, 2.9e9), (1500, 2.1e9), (600, 9e8)])
def test_contribution_to_wide_grids(bins, bandwidth):
    """H of one redone path, bin by bin.  A seed is within 2e-7 rad (phase rounded to FP32) and 1e-7 (sine, cosine) of its place, each of the
    at most 16 rotations from it within 2e-7 rad of its angle (rounded to FP32) and 2e-7 (its sine and cosine, the product): 7e-6."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    fg, tg = I.FreqGrid(28e9, bandwidth, bins), I.TimeGrid(0.0, 1e-8, 3)
    f = fg.fc - 0.5 * bandwidth + bandwidth / bins * np.arange(bins)
    with drt.Context(0) as ctx:
        for seed in range(2, 14):
            link = ctx.load(plates(1, seed), I.chains_to_pathset([[(I.T_R, 0)]]))
            r = {k: v.cpu().numpy() for k, v in link.extrapolate(tg, fg, drt.FP64).items() if v is not None}
            a = r["amp"][..., 0] + 1j * r["amp"][..., 1]
            x = r["tau"][:, :, None] * f
            want = (a[:, :, None] * np.exp(-2j * np.pi * (x - np.floor(x))))[:, 0]
            H = torch.full((tg.n_steps, bins), float("nan"), dtype=torch.complex64, device="cuda")
            with ctx.batch([link], [tg], [fg], [H]) as b:
                b.run()
                assert b.info(redo=True)["redo_steps"] == tg.n_steps
            assert (np.abs(H.cpu().numpy() - want) <= 7e-6 * np.abs(a)).all()
            link.unload()
