"""Tables whose systems are singular: interpolation weights may be infinite or not
numbers.  On the CPU, the order that ranks a row's weights gives every position
a rank of its own; on the GPU, such a game ends with a status and leaves the
solver as good as new."""
import os
import subprocess

import numpy as np
import pytest

from test_gpu_amg_paths import band_game

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1107_1653_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "weight_order.h"
int main() {
    const double val[] = {NAN, -NAN, INFINITY, -INFINITY, 0.0, -0.0, 1.0, 1.0, -2.0};
    const int V = sizeof val / sizeof *val;
    long rows = 0, bad = 0, order = 0;
    for (int m = 1; m <= 5; ++m) {
        int n = 1;
        for (int k = 0; k < m; ++k) n *= V;
        for (int code = 0; code < n; ++code) {
            double w[5];
            for (int k = 0, c = code; k < m; ++k, c /= V) w[k] = val[c % V];
            unsigned seen = 0;
            for (int q = 0; q < m; ++q) {
                int rank = 0;
                for (int t = 0; t < m; ++t) {
                    rank += gs::weight_before(w[t], t, w[q], q);
                    order += w[t] > w[q] && !gs::weight_before(w[t], t, w[q], q);
                }
                seen |= 1u << rank;
            }
            ++rows;
            bad += seen != (1u << m) - 1;
        }
    }
    std::printf("%ld %ld %ld\n", rows, bad, order);
}
"""


def test_every_position_has_a_rank_of_its_own(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    rows, bad, order = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert rows == sum(9 ** m for m in range(1, 6)) and bad == 0 and order == 0


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("theta", [0.0, 1e-12])
def test_game_without_exit(gs, theta, prec):
    """A ring that is never left, undiscounted: every system is singular."""
    n = 900
    rng = np.random.default_rng(4)
    col = (np.arange(n)[:, None, None] + np.array([-2, -1, 1, 3])[None, None, :]) % n
    col = np.repeat(col, 4, axis=1).reshape(-1).astype(np.int32)
    prob = rng.dirichlet(np.ones(4), size=4 * n).reshape(-1)
    prob[::4] *= 1e-14
    prob = (prob.reshape(-1, 4) / prob.reshape(-1, 4).sum(axis=1, keepdims=True)).reshape(-1)
    rp = np.arange(4 * n + 1, dtype=np.int64) * 4
    rew = rng.uniform(-1, 1, 4 * n)
    good = band_game(n, 3, 5)
    with gs.GameSolver(precision=prec, game_solver=1, amg_theta=theta, max_outer=5, max_inner=5) as s:
        s.set_game(n, 2, 2, *good, 0.995)
        s.solve(allow_notconv=True)
        v = s.get_value()
        s.set_game(n, 2, 2, rp, col, prob, rew, 1.0)
        # (in float64 rounding can leave the last pivot small but not zero: a value
        # of 1e16 whose relative residual is within the tolerance)
        assert gs.gamesolve_solve(s.h, None) in (gs.GS_OK, gs.GS_ENOTCONV, gs.GS_EINVAL)
        s.set_game(n, 2, 2, *good, 0.995)
        s.solve(allow_notconv=True)
        assert np.array_equal(s.get_value(), v)
