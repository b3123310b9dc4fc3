"""The tables path's multigrid at the edges of its kernels, against the float64
oracle: rows narrower and wider than a warp, couplings to many neighbours (many
smoother colours), games at and just above the size that is inverted directly,
levels on either side of the one-block limit.  Bars as in test_gpu_amg.
"""
import numpy as np
import pytest

import oracle
from oracle.game import game_from_csr

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-10, "mixed": 1e-9}


def band_game(n, b, seed):
    """States on a line, moves to the b neighbours on either side (those outside
    leave the game) with random weights that fall with the distance; 2 x 2
    actions, one of MAX's a stop (an empty row)."""
    rng = np.random.default_rng(seed)
    rp, col, prob, rew = [0], [], [], []
    for x in range(n):
        for a in range(2):
            for _ in range(2):
                if a == 1 and x % 7 == 0:
                    rp.append(len(col))
                    rew.append(rng.uniform(-1, 1))
                    continue
                d = np.array([k for k in range(-b, b + 1) if k != 0])
                w = rng.uniform(0.5, 1.0, len(d)) / np.abs(d)
                w /= w.sum()
                y = x + d
                ok = (y >= 0) & (y < n)
                col.extend(y[ok].tolist())
                prob.extend(w[ok].tolist())
                rp.append(len(col))
                rew.append(rng.uniform(-0.01, 0.01))
    return np.array(rp, np.int64), np.array(col, np.int32), np.array(prob), np.array(rew)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("coarsening", [0, 1])
@pytest.mark.parametrize("n,b", [(40, 1), (128, 3), (129, 3), (129, 20), (700, 1), (700, 20), (1500, 6), (2049, 2), (2300, 31)])
def test_band_games(gs, n, b, coarsening, prec):
    mu = 0.995
    rp, col, prob, rew = band_game(n, b, 7 * n + b)
    game = game_from_csr(n, 2, 2, rp, col, prob, rew, mu)
    ref = oracle.policy_iteration(game)
    with gs.GameSolver(precision=prec, game_solver=1, amg_coarsening=coarsening) as s:
        s.set_game(n, 2, 2, rp, col, prob, rew, mu)
        st = s.solve()
        v = s.get_value()
        a, bb = s.get_policy()
    assert st["converged"] == 1
    assert np.max(np.abs(v - ref.v)) / np.max(np.abs(ref.v)) <= TOL[prec], st
    sure = ref.gap_max > 1e-8
    assert np.array_equal(a[sure], ref.alpha[sure])
    sure_b = ref.gap_min > 1e-8
    assert np.array_equal(bb.reshape(ref.beta.shape)[sure_b], ref.beta[sure_b])
