"""What needed no more than an HBM budget without two-float numbers needs no more with them: their copies of a link's arrays and the ray
tracer's scratch give way.  The smallest budget is that of the same scene with a material (of no face) that rules them out."""
import dataclasses
import os

import numpy as np
import pytest

from paper_2205_00237_gb300 import inputs as I

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")
TG, FG = I.TimeGrid(0.0, 2e-3, 40), I.FreqGrid(60e9, 1e9, 16)


def retraced(drt, ctx, scene, paths):
    return ctx.load(scene, paths).synthesize_H_retraced(TG, FG, [0, 20], 2, with_tiles=True, precision=drt.FP64)


def traced_first(drt, ctx, scene, paths):
    link = ctx.load(scene, paths)
    link.trace_paths(0.0, 2, with_tiles=True)
    return link.synthesize_H(TG, I.FreqGrid(60e9, 1e9, 16), drt.FP64)


def one_call(drt, ctx, scene, paths):
    return ctx.load(scene, paths).synthesize_H(TG, FG, drt.FP64)


def bulk_call(drt, ctx, scene, paths):
    return ctx.load(scene, paths).synthesize_H(TG, FG, drt.FP32_BULK)


def two_links(drt, ctx, scene, paths):
    links = [ctx.load(scene, paths) for _ in range(2)]
    links[1].synthesize_H(TG, FG, drt.FP64)
    return links[0].synthesize_H(TG, FG, drt.FP64)


def batch(drt, ctx, scene, paths):
    import torch
    H = torch.empty(TG.n_steps, FG.n_bins, dtype=torch.complex64, device="cuda")
    with ctx.batch([ctx.load(scene, paths)], [TG], [FG], [H]) as b:
        b.run()
        torch.cuda.synchronize()
    return H


def unloaded(drt, ctx, scene, paths):
    """A link loaded and unloaded before: its blocks are pooled."""
    ctx.load(scene, paths).unload()
    return ctx.load(scene, paths.subset(np.arange(40))).synthesize_H(TG, FG, drt.FP64)


@pytest.mark.parametrize("call", [retraced, traced_first, one_call, bulk_call, two_links, batch, unloaded])
def test_smallest_budget(call):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    scene, paths = I.scene_canyon(0), I.PathSet.from_npz(os.path.join(GOLD, "pathset_canyon_seed0.npz"))
    extra = scene.materials[:1].copy()
    extra["eps_r"] = 2e6
    lean = dataclasses.replace(scene, materials=np.concatenate([scene.materials, extra]))

    def run(sc, budget):
        with drt.Context(0, hbm_budget=budget) as ctx:
            try:
                return call(drt, ctx, sc, paths).cpu()
            except drt.DrtError as e:
                assert e.code == drt.DRT_ENOMEM
                return None

    lo, hi = 1 << 16, 1 << 28
    want = run(lean, hi)
    while hi - lo > 4096:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if run(lean, mid) is not None else (mid, hi)
    got = run(scene, hi)
    assert got is not None and float(torch.linalg.vector_norm(got - want)) <= 1e-4 * float(torch.linalg.vector_norm(want))
