"""Which pass a ray-tracing run takes: FP64 alone in scenes of few faces, two-float numbers first in the others; and what the latter finds
where bodies have turned."""
import os

import pytest

import host_program
from paper_2205_00237_gb300 import inputs as I
from test_two_float_range import ctx, spun  # noqa: F401

GOLD = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")

RULE = """
#include <cstdio>
#include "drt_internal.h"
// in: faces, edges, tiles, order; out: whether the two-float passes run
int main() {
    double f, e, t, o;
    while (std::scanf("%lf %lf %lf %lf", &f, &e, &t, &o) == 4) {
        drt::LinkDev L{};
        L.n_faces = (int)f;
        L.n_edges = (int)e;
        L.n_tiles = (int)t;
        std::printf("%d\\n", (int)drt::trace_two_float(L, (int)o, L.n_tiles > 0));
    }
}
"""


def test_rule(tmp_path):
    cases = [((7, 12, 0, 0), 0), ((7, 12, 0, 1), 0), ((7, 12, 0, 2), 0), ((31, 84, 714, 2), 0), ((89, 216, 3875, 2), 1),
             ((30, 0, 0, 0), 0), ((31, 0, 0, 0), 1), ((10, 0, 0, 1), 0), ((11, 0, 0, 1), 1), ((40, 0, 0, 2), 0), ((41, 0, 0, 2), 1),
             ((1, 0, 16382, 1), 0), ((1, 0, 16383, 1), 1), ((1, 126, 0, 2), 0), ((1, 127, 0, 2), 1), ((0, 0, 0, 0), 0)]
    got = host_program.run(host_program.build(RULE, tmp_path), [c for c, _ in cases])
    assert [int(g[0]) for g in got] == [w for _, w in cases]


@pytest.mark.gpu
@pytest.mark.parametrize("w0,t,order", [(0.9, 0.6, 1), (40.0, 1.3, 1), (40.0, 1.3, 2)])
def test_turned_bodies(ctx, w0, t, order):  # noqa: F811
    from test_gpu_trace import compare_rays
    scene = spun(I.scene_canyon(0), w0)
    link = ctx.load(scene, I.PathSet.from_npz(os.path.join(GOLD, "pathset_canyon_seed0.npz")))
    compare_rays(link.trace_paths(t, order, with_tiles=False), scene, t, order, False)
    link.unload()
