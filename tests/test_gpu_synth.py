"""H synthesis at the edges of its tiles: bin counts around 16, 128, 256 and 512 (the tile widths), path counts around the
16 paths of a matrix step, step counts that select one, four and eight warps per tile; single-link and batched.

Reference: the library's own FP64 records (delay and amplitude) summed term by term in FP64.  Bar: a term's error is at
most ~4e-7 for each of the two or three hardware sines and cosines it is a product of, 2e-7 for the rounding of the
record's phase, 2.4e-7 for the 22-bit operands and ~1e-6 for the FP32 additions, below 4e-6 |a_p| in all, so a bin's is below
4e-6 sum |a_p|.  The batch runs the FP32-bulk form, whose phases are within 1e-3 rad: 1e-3 sum |a_p|.
"""
import os

import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")
PATHS = [0, 1, 2, 15, 16, 17, 33, 65, 400]


@pytest.fixture(scope="module")
def loaded():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    scene = I.scene_link(1)
    paths = I.PathSet.from_npz(os.path.join(GOLD, "pathset_link_seed1.npz"))
    with drt.Context(0) as ctx:
        yield drt, ctx, [ctx.load(scene, paths.subset(np.arange(p))) for p in PATHS]


def direct(drt, link, tg, fg):
    """(H, sum of |a|) per instant from the link's FP64 records."""
    r = {k: v.cpu().numpy() for k, v in link.extrapolate(tg, fg, drt.FP64).items() if v is not None}
    a = np.where(r["flags"] == 0, r["amp"][..., 0] + 1j * r["amp"][..., 1], 0)
    tau = np.where(r["flags"] == 0, r["tau"], 0.0)   # a step that is no ray may have no delay
    f = fg.fc - 0.5 * fg.bandwidth + fg.bandwidth / fg.n_bins * np.arange(fg.n_bins)
    x = tau[:, :, None] * f
    return (a[:, :, None] * np.exp(-2j * np.pi * (x - np.floor(x)))).sum(1), np.abs(a).sum(1)


@pytest.mark.parametrize("bins", [1, 16, 17, 127, 129, 255, 257, 512, 513, 1025, 4096])
def test_bins(loaded, bins):
    drt, ctx, links = loaded
    fg = I.FreqGrid(28e9, 400e6, bins)
    for i, T in ((8, 7), (4, 33), (1, 3)):
        tg = I.TimeGrid(0.2, 1e-3, T)
        ref, bar = direct(drt, links[i], tg, fg)
        H = links[i].synthesize_H(tg, fg, drt.FP64).cpu().numpy()
        assert (np.abs(H - ref) <= 4e-6 * bar[:, None]).all()


@pytest.mark.parametrize("steps", [5, 1300, 2600])   # eight, four and one warp per tile (where paths allow)
def test_paths(loaded, steps):
    drt, ctx, links = loaded
    tg, fg = I.TimeGrid(0.0, 1e-4, steps), I.FreqGrid(28e9, 400e6, 40)
    for link in links:
        ref, bar = direct(drt, link, tg, fg)
        H = link.synthesize_H(tg, fg, drt.FP64).cpu().numpy()
        assert (np.abs(H - ref) <= 4e-6 * bar[:, None]).all()


@pytest.mark.parametrize("bins", [1, 128, 300, 512, 513])
def test_batch(loaded, bins):
    import torch
    drt, ctx, links = loaded
    fg = I.FreqGrid(28e9, 400e6, bins)
    tgs = [I.TimeGrid(0.1, 1e-3, 1 + 13 * i) for i in range(len(links))]
    Hs = [torch.full((t.n_steps, bins), float("nan"), dtype=torch.complex64, device="cuda") for t in tgs]
    with ctx.batch(links, tgs, [fg] * len(links), Hs) as b:
        b.run()
        torch.cuda.synchronize()
    for link, tg, H in zip(links, tgs, Hs):
        ref, bar = direct(drt, link, tg, fg)
        assert (np.abs(H.cpu().numpy() - ref) <= 1e-3 * bar[:, None]).all()
