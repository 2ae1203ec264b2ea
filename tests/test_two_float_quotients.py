"""Two-float quotients at the end of the FP32 range, where 1 / x is 0 (x from 2^126 on): metals at low carriers, whose Fresnel
coefficients divide by |eps_c| and its square, and long chains, whose spreading divides by a product of ten lengths."""
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
// in: sigma, fc; out: whether two-float numbers apply to a scene of that metal
int main() {
    double sigma, fc;
    while (std::scanf("%lf %lf", &sigma, &fc) == 2) {
        drt_scene s{};
        drt_body b{};
        drt_material m[2]{};
        b.k[2] = 1.0;
        m[0].eps_r = m[1].eps_r = 1.0;
        m[1].sigma = sigma;
        s.bodies = &b;
        s.materials = m;
        s.n_bodies = 1;
        s.n_materials = 2;
        drt_path_set ps{};
        drt::PackedLink H;
        if (drt::pack_link(&s, &ps, H)) return 1;
        const drt_time_grid tg{0.0, 1e-3, 10, 0};
        drt_freq_grid fg{};
        fg.fc = fc;
        fg.n_bins = 1;
        std::printf("%d\\n", (int)drt::ff_applies(H.view, tg, fg));
    }
}
"""


def test_rule(tmp_path):
    """sigma / (2 pi fc eps0) up to 1e15: 1.8e18 Hz / fc for 1e8 S/m."""
    cases = [((0, 1.0), 1), ((0.1, 1.0), 1), ((6e7, 2e5), 1), ((6e7, 1.1e3), 1), ((6e7, 1.0e3), 0), ((6e7, 1.0), 0),
             ((1e8, 1e9), 0), ((99e6, 1.8e3), 1), ((99e6, 1.7e3), 0)]
    got = host_program.run(host_program.build(RULE, tmp_path), [c for c, _ in cases])
    assert [int(g[0]) for g in got] == [w for _, w in cases]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2205_00237_gb300 import drt
    with drt.Context(0) as c:
        yield c


def compare(ctx, scene, paths, tg, fg):
    """H within 1e-6 sum |a_p| of the FP64 kernels': the rounding of the records."""
    import torch
    from paper_2205_00237_gb300 import drt
    link = ctx.load(scene, paths)
    H = link.synthesize_H(tg, fg, drt.FP64)
    want = torch.full_like(H, float("nan"))
    link.synthesize_H_noalloc(tg, fg, want)
    r = link.extrapolate(tg, fg, drt.FP64)
    mag = torch.where(r["flags"] == 0, torch.linalg.vector_norm(r["amp"], dim=-1), torch.zeros_like(r["tau"]))
    link.unload()
    assert bool(mag.sum() > 0) and bool(((H - want).abs() <= 1e-6 * mag.sum(1, keepdim=True)).all())


@pytest.mark.gpu
@pytest.mark.parametrize("sigma,fc", [(6e7, f) for f in (2e5, 1e5, 7e4, 6e4, 5e4, 4.5e4, 4e4, 3e4, 2e4, 1e4, 1.1e3, 1.0)])
def test_metals_at_low_carriers(ctx, sigma, fc):
    """A ground of copper seen at cos = 0.13: the product of the two divisors passes 2^126 between 62 and 39 kHz, then 2^128."""
    scene = I.scene_tiny(0)
    mats = scene.materials.copy()
    mats["sigma"][0] = sigma
    paths = I.PathSet.from_npz(os.path.join(GOLD, "pathset_tiny_seed0.npz"))
    compare(ctx, dataclasses.replace(scene, materials=mats), paths, I.TimeGrid(0.0, 1e-2, 70), I.FreqGrid(fc, 0.1 * fc, 20))


@pytest.mark.gpu
@pytest.mark.parametrize("leg", [5000.0, 6324.0, 6900.0, 9000.0])
def test_long_tile_chains(ctx, leg):
    """Four tiles between five legs: the spreading's divisor leg^10 passes 2^126 at 6211 m, and 2^128 at 7134 m."""
    scene = I.scene_link(0)
    tiles = np.repeat(scene.tiles[:1], 4)
    x = leg * np.array([0.3, 0.6, 0.9, 1.2])
    y = np.array([0.0, 1.0, 0.0, 1.0]) * np.sqrt(1 - 0.09) * leg
    for i in range(4):
        tiles[i]["c"] = [x[i], y[i], 0.0]
        tiles[i]["n"] = [0.0, 1.0 if i % 2 == 0 else -1.0, 0.0]
    tiles["body"], tiles["area"] = 0, 1e6
    tx, rx = scene.tx.copy(), scene.rx.copy()
    tx["r"], rx["r"] = [0.0, y[1], 0.0], [1.5 * leg, 0.0, 0.0]
    tx["v"], rx["v"] = [3.0, 0.0, 1.0], [-5.0, 0.0, 2.0]
    paths = I.chains_to_pathset([[(I.T_S, 0), (I.T_S, 1), (I.T_S, 2), (I.T_S, 3)]])
    compare(ctx, dataclasses.replace(scene, tiles=tiles, tx=tx, rx=rx), paths, I.TimeGrid(0.0, 1e-2, 40),
            I.FreqGrid(1e6, 1e5, 20))
