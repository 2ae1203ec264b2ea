"""The ray tracer's two-float pass, which discards pairs in FP32 first, against FP64 on random candidates close to grazing, and its
segment-face tests on the segments of the rays among them.  On the CPU."""
import os

import pytest

import host_program

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def trace(tmp_path_factory):
    with open(os.path.join(HERE, "two_float_tracing.cu")) as f:
        exe = host_program.build(f.read(), tmp_path_factory.mktemp("trace"))
    return lambda *q: [int(x) for x in host_program.run(exe, [q])[0]]


@pytest.mark.parametrize("most_d,extent,shortest,angle,come_from,margin,least", [
    (2, 20, 1, 0.2, 0, 1e-13, 0.7), (1, 500, 0.01, 1e-2, 0, 1e-13, 0.6), (1, 20, 1e-4, 1e-7, 0, 1e-13, 0.3),
    (2, 500, 0.01, 1e-4, 0, 1e-13, 0.4), (2, 20, 1, 0.2, 1e4, 1e-13, 0.5),
    # margins far above the FP32 error at angles where the points' error is amplified most
    (2, 500, 50, 3e-3, 0, 0.5, 0.8), (2, 100, 10, 1e-3, 0, 0.3, 0.8), (0, 500, 100, 1e-3, 0, 0.9, 0.9)])
def test_candidates(trace, most_d, extent, shortest, angle, come_from, margin, least):
    """(least: the share that is decided without FP64.)  FP64's own solve may fail by a chance of its line search: 1 in 10000."""
    n, decided, rays, wrong, unconverged, pairs, sure, differ, dropped, off, near = trace(
        most_d, extent, shortest, angle, come_from, margin, 21, 30000)
    assert wrong == 0 and unconverged <= n // 10000 and rays > 1000 and decided > least * n
    assert differ == 0 and sure > 0.3 * pairs
    assert off == 0 and near == 0 and (dropped > 100 or margin < 0.1)
