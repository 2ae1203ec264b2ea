"""Where two-float numbers may be used when bodies rotate: an angle has the same 47 bits as a length, so a turn of A rad at the distance R
costs what a coordinate of A R does, and past a few thousand rad the whole turns are not taken off any more.  Such calls
run in FP64."""
import dataclasses
import os

import numpy as np
import pytest

import host_program
from paper_2205_00237_gb300 import inputs as I

GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")

RULE = """
#include <cstdio>
#include "drt_internal.h"
// in: w0, wdot (rad/s, rad/s^2) of a body at rest 3 m from the origin, t_start, dt, n_steps, fc; out: whether two-float applies
int main() {
    double w0, wdot, t0, dt, n, fc;
    while (std::scanf("%lf %lf %lf %lf %lf %lf", &w0, &wdot, &t0, &dt, &n, &fc) == 6) {
        drt_scene s{};
        drt_body b{};
        b.o[0] = 3.0;
        b.k[2] = 1.0;
        b.w0 = w0;
        b.wdot = wdot;
        s.bodies = &b;
        s.n_bodies = 1;
        s.rx.r[0] = 100.0;   // the scene's extent
        drt_path_set ps{};
        drt::PackedLink H;
        if (drt::pack_link(&s, &ps, H)) return 1;
        const drt_time_grid tg{t0, dt, (int)n, 0};
        drt_freq_grid fg{};
        fg.fc = fc;
        fg.n_bins = 1;
        std::printf("%d\\n", (int)drt::ff_applies(H.view, tg, fg));
    }
}
"""


def test_rule(tmp_path):
    """100 m of extent at 60 GHz leaves 12 rad below 2^18 wavelengths (1310 m); at 100 MHz the cap of 4096 rad decides."""
    exe = host_program.build(RULE, tmp_path)
    cases = [((0, 0, 0, 1e-3, 10, 60e9), 1), ((0, 0, 1.7e9, 1e-3, 10, 60e9), 1),
             ((11.9, 0, 0, 0.1, 10, 60e9), 1), ((12.3, 0, 0, 0.1, 10, 60e9), 0), ((-12.3, 0, 0, 0.1, 10, 60e9), 0),
             ((12.3, 0, 0, 0.09, 10, 60e9), 1), ((12.3, 0, -1.0, 0.05, 10, 60e9), 0),
             ((0, 23.8, 0, 0.1, 10, 60e9), 1), ((0, 24.6, 0, 0.1, 10, 60e9), 0),
             ((0.3, 0, 1.7e9, 1e-3, 10, 60e9), 0), ((1.0, 0, 3e7, 1e-3, 10, 60e9), 0),
             ((4095, 0, 0, 0.1, 10, 1e8), 1), ((4097, 0, 0, 0.1, 10, 1e8), 0), ((4097, 0, 0, 0.1, 10, 1.0), 0),
             ((1e300, 0, 1e300, 0.1, 10, 1.0), 0), ((0, 1e300, 1e300, 0.1, 10, 1.0), 0)]
    got = host_program.run(exe, [c for c, _ in cases])
    assert [int(g[0]) for g in got] == [w for _, w in cases]


def spun(scene, w0, wdot=0.0):
    bodies = scene.bodies.copy()
    bodies["w0"][1:], bodies["wdot"][1:] = w0, wdot
    bodies["v"][1:] = 0.0
    rx = scene.rx.copy()   # nothing moves but by rotation, whatever the instant
    rx["v"] = 0.0
    return dataclasses.replace(scene, bodies=bodies, rx=rx)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    with drt.Context(0) as c:
        yield c


def both(ctx, scene, tg, fg):
    """H of the FP64 form, of the FP64 kernels, and sum |a_p| of the FP64 records."""
    import torch
    from paper_2205_00237_gb300 import drt
    link = ctx.load(scene, I.PathSet.from_npz(os.path.join(GOLD, "pathset_tiny_seed0.npz")))
    H = link.synthesize_H(tg, fg, drt.FP64)
    want = torch.full_like(H, float("nan"))
    link.synthesize_H_noalloc(tg, fg, want)
    r = link.extrapolate(tg, fg, drt.FP64)
    mag = torch.linalg.vector_norm(r["amp"], dim=-1)
    link.unload()
    return H, want, torch.where(r["flags"] == 0, mag, torch.zeros_like(mag)).sum(1, keepdim=True)


@pytest.mark.gpu
@pytest.mark.parametrize("turns", [3, 30, -30])
def test_turned_bodies(ctx, turns):
    """Bar: 1e-6 sum |a_p|, the rounding of the records (phases of both forms within 2e-7 rad, amplitudes within 6e-8)."""
    w = 2 * np.pi * turns
    tg, fg = I.TimeGrid(0.9, 1e-3, 100), I.FreqGrid(1e9, 1e8, 40)
    H, want, mag = both(ctx, spun(I.scene_tiny(0), w), tg, fg)
    assert bool(((H - want).abs() <= 1e-6 * mag).all()) and bool(mag.max() > 0)


@pytest.mark.gpu
@pytest.mark.parametrize("w0,wdot,t", [(5000.0, 0.0, 1.0), (0.0, 9000.0, 1.0), (0.3, 0.0, 1.7e8), (1e4, 0.0, 1e4)])
def test_beyond_the_range_is_fp64(ctx, w0, wdot, t):
    import torch
    H, want, mag = both(ctx, spun(I.scene_tiny(0), w0, wdot), I.TimeGrid(t, 1e-5, 64), I.FreqGrid(28e9, 4e8, 20))
    assert torch.equal(H, want) and bool(mag.max() > 0)


@pytest.mark.gpu
@pytest.mark.parametrize("w0,t", [(0.9, 0.6), (40.0, 1.3), (0.3, 1e8)])
def test_traced_rays_of_turned_bodies(ctx, w0, t):
    from test_gpu_trace import compare_rays
    scene = spun(I.scene_tiny(0), w0)
    link = ctx.load(scene, I.PathSet.from_npz(os.path.join(GOLD, "pathset_tiny_seed0.npz")))
    compare_rays(link.trace_paths(t, 2, with_tiles=False), scene, t, 2, False)
    link.unload()
