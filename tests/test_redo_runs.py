"""Which warp takes which steps of a redo list: every step once, and the runs spread over the warps, also where all of them start at
multiples of 32 (paths that are redone at every step)."""
import pytest

import host_program

PROGRAM = """
#include <algorithm>
#include <cstdio>
#include <vector>
#include "drt_physics.cuh"
// in: runs of `len` steps, their number, warps; out: steps taken a time other than once, the most runs of a warp, warps' stride
int main() {
    double len, n, w;
    while (std::scanf("%lf %lf %lf", &len, &n, &w) == 3) {
        const int L = (int)len, total = L * (int)n, warps = (int)w;
        std::vector<int4> items(total);
        for (int k = 0; k < total; ++k) items[k] = make_int4(0, 0, k, L << 8 | k % L);
        int count = total;
        const drt::RedoList list{&count, items.data(), total};
        std::vector<int> taken(total, 0);
        int most = 0, wrong = 0;
        for (int warp = 0; warp < warps; ++warp) {
            int steps = 0;
            for (int lane = 0; lane < 32; ++lane)
                drt::for_redo_runs(list, warp, warps, lane, [&](int k, int4 it) {
                    ++taken[k];
                    ++steps;
                    wrong += it.z != k;
                });
            most = std::max(most, steps / L);
        }
        for (int t : taken) wrong += t != 1;
        std::printf("%d %d %d\\n", wrong, most, drt::redo_stride(warps));
    }
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    return host_program.build(PROGRAM, tmp_path_factory.mktemp("runs"))


@pytest.mark.parametrize("warps", [1, 2, 31, 32, 33, 1184, 1216, 2432])
@pytest.mark.parametrize("length", [1, 4, 16, 32])
def test_runs_are_spread(program, length, warps):
    for n in (1, 40, 800, 3000):
        wrong, most, stride = host_program.run(program, [[length, n, warps]])[0]
        assert wrong == 0 and warps - 1 <= stride <= warps
        assert most <= -(-n // int(stride)) + 1
