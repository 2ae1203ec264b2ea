"""H of the FP64 form, whose records are computed in two-float numbers with an FP64 step for what those cannot decide, against
the same call on the FP64 kernels (drt_synthesize_H_noalloc, which keeps them).

Bar: both round the amplitude and the phase seed of a path to FP32 (6e-8 and 3e-8 turns = 2e-7 rad, possibly to neighbouring
values), and the two-float phase is within 2^-46 of 2^21 wavelengths = 2e-7 rad, so a bin differs by less than 1e-6 sum |a_p|;
sum |a_p| comes from the FP64 records.  A path whose validity differed would show with its whole amplitude.
"""
import dataclasses
import math
import os

import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


def base(name, k):
    scene = {"tiny": I.scene_tiny, "link": I.scene_link, "canyon": I.scene_canyon}[name](k)
    return scene, I.PathSet.from_npz(os.path.join(GOLD, f"pathset_{name}_seed{k}.npz"))


def with_wedges(scene, seed):
    """The scene with every other wedge at an interior angle of its own (n between 1.1 and 1.95)."""
    rng = np.random.default_rng(seed)
    edges = scene.edges.copy()
    for e in edges[::2]:
        n = rng.uniform(1.1, 1.95)
        t = np.cross(e["b"] - e["a"], e["n0"])
        e["nn"] = math.cos((n - 1) * math.pi) * e["n0"] + math.sin((n - 1) * math.pi) * t / np.linalg.norm(t)
        e["wedge_n"] = n
    return dataclasses.replace(scene, edges=edges)


def spinning(scene):
    bodies = scene.bodies.copy()
    bodies["wdot"][1:] = 0.7
    bodies["w0"][1:] = -1.3
    return dataclasses.replace(scene, bodies=bodies)


def compare(scene, paths, tg, fg):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    with drt.Context(0) as ctx:
        link = ctx.load(scene, paths)
        H = link.synthesize_H(tg, fg, drt.FP64)
        want = torch.full_like(H, float("nan"))
        link.synthesize_H_noalloc(tg, fg, want)
        r = link.extrapolate(tg, fg, drt.FP64)
        mag = torch.linalg.vector_norm(r["amp"], dim=-1)
        bar = 1e-6 * torch.where(r["flags"] == 0, mag, torch.zeros_like(mag)).sum(1, keepdim=True)
        valid = int((r["flags"] == 0).sum())
        assert bool(((H - want).abs() <= bar).all()), float(((H - want).abs() / (bar + 1e-30)).max())
        link.unload()
    return valid


@pytest.mark.parametrize("name,k", [("tiny", 0), ("tiny", 1), ("link", 0), ("link", 3), ("canyon", 0)])
@pytest.mark.parametrize("t_start", [0.0, -0.75])
def test_workloads(name, k, t_start):
    scene, paths = base(name, k)   # link 0 has a chain with a tile in the plane of its edge's wedge face: decided in FP64
    fc = 60e9 if name == "canyon" else 28e9
    assert compare(scene, paths, I.TimeGrid(t_start, 1.7e-3, 333), I.FreqGrid(fc, 400e6, 40)) > 0


def test_wedges_of_any_angle_and_rotation():
    scene, paths = base("canyon", 0)
    fg = I.FreqGrid(60e9, 1e9, 33)
    assert compare(with_wedges(scene, 1), paths, I.TimeGrid(0.0, 2e-3, 200), fg) > 0
    assert compare(spinning(scene), paths, I.TimeGrid(0.0, 3e-3, 500), fg) > 0


@pytest.mark.parametrize("lengths", [(1,), (2,), (3,), (4,)])
def test_random_chains(lengths):
    """Chains that are mostly no rays: every decision counts; 4 vertices and several diffractions among them."""
    rng = np.random.default_rng(sum(lengths))
    scene, _ = base("canyon", 0)
    paths = I.draw_chains_batch(rng, scene, 1500, p_r=0.5, lengths=lengths)
    compare(scene, paths, I.TimeGrid(0.0, 0.05, 20), I.FreqGrid(28e9, 200e6, 20))


def test_large_scene_keeps_fp64():
    """Coordinates beyond 2^18 wavelengths: the records come from the FP64 kernels, bit for bit those of the other call."""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    scene, paths = base("tiny", 0)
    far = dataclasses.replace(scene, tx=scene.tx.copy(), rx=scene.rx.copy())
    far.rx["r"] = far.rx["r"] + [2e6, 0, 0]
    tg, fg = I.TimeGrid(0.0, 1e-3, 50), I.FreqGrid(60e9, 1e8, 20)
    with drt.Context(0) as ctx:
        link = ctx.load(far, paths)
        H = link.synthesize_H(tg, fg, drt.FP64)
        want = torch.empty_like(H)
        link.synthesize_H_noalloc(tg, fg, want)
        assert bool(H.abs().max() > 0) and torch.equal(H, want)


@pytest.mark.parametrize("name,k", [("link", 0), ("link", 1), ("link", 2), ("link", 3), ("canyon", 0)])
def test_doppler_of_redone_steps(name, k):
    """The FP32-bulk records' redone steps (their delay is the FP64 one to 1e-12; an FP32 step's is within 1e-9 of it, but for the first
    step of a chunk, a multiple of 4, whose delay is an FP64 anchor while its Doppler shift is FP32) have the FP64 Doppler shift to FP32 rounding, also where a point of a chain that is no ray runs at a good part of the speed of light: 1e-6
    covers the rounding of the result and of the velocities (2^-40)."""
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    scene, paths = base(name, k)
    tg, fg = I.TimeGrid(0.0, 1e-3, 1237), I.FreqGrid(60e9 if name == "canyon" else 28e9, 400e6, 1)
    with drt.Context(0) as ctx:
        link = ctx.load(scene, paths)
        a = {q: v.cpu().numpy() for q, v in link.extrapolate(tg, fg, drt.FP64).items() if v is not None}
        b = {q: v.cpu().numpy() for q, v in link.extrapolate(tg, fg, drt.FP32_BULK).items() if v is not None}
    fine = (a["flags"] & 24) == 0   # converged and not degenerate
    redone = fine & (np.abs(b["tau"] / a["tau"] - 1) < 1e-12) & (a["flags"] == b["flags"])
    redone[::4] = False
    assert redone.any()
    err = np.abs(b["doppler"] - a["doppler"])[redone]
    # a step of FP32 geometry whose delay agrees by chance keeps the FP32 form's 0.1 Hz
    assert (err <= np.maximum(1e-6 * np.abs(a["doppler"][redone]), 0.1)).all(), err.max()
