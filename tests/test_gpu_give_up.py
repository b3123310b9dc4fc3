"""Waits that give up inside a solve: the call ends with GS_ETIMEOUT, what it leaves
behind is what was there before, and the solver's next call is unharmed."""
import numpy as np
import pytest

from test_gpu_amg_paths import band_game

pytestmark = pytest.mark.gpu


def give_up(gs, s, on):
    assert gs.gamesolve_selftest_give_up(s.h, on) == gs.GS_OK


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("opts", [{}, {"amg_coarsening": 1}, {"fmg": 1}])
def test_tables_setup(gs, opts, prec):
    """Splitting and colouring end early and leave points undecided."""
    n = 2300
    rp, col, prob, rew = band_game(n, 6, 5)
    with gs.GameSolver(precision=prec, game_solver=1, **opts) as s:
        s.set_game(n, 2, 2, rp, col, prob, rew, 0.995)
        s.solve()
        v = s.get_value()
        for _ in range(3):
            give_up(gs, s, 1)
            with pytest.raises(gs.GameSolveError) as e:
                s.solve()
            assert e.value.status == gs.GS_ETIMEOUT
            give_up(gs, s, 0)
            s.solve()
            assert np.array_equal(s.get_value(), v)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("opts", [{}, {"cycle_kernel": 1}])
@pytest.mark.parametrize("side,variant", [(127, 0), (255, 1)])
def test_isaacs_policies_stay(gs, side, variant, opts, prec):
    """No reply is improved at a value whose evaluation was given up."""
    n, m1 = side * side, 5 if variant else 4
    rng = np.random.default_rng(side)
    v0 = rng.uniform(-1, 1, n)
    alpha0 = rng.integers(0, m1, n).astype(np.uint8)
    beta0 = rng.integers(0, 4, (n, m1)).astype(np.uint8)
    with gs.GameSolver(precision=prec, **opts) as s:
        s.set_isaacs_grid(side, variant, 3)
        s.set_initial(v0, alpha0, beta0)
        s.solve()
        v = s.get_value()
        s.set_initial(v0, alpha0, beta0)
        give_up(gs, s, 1)
        with pytest.raises(gs.GameSolveError) as e:
            s.solve()
        assert e.value.status == gs.GS_ETIMEOUT
        alpha, beta = s.get_policy()
        assert np.array_equal(alpha, alpha0) and np.array_equal(beta, beta0)
        give_up(gs, s, 0)
        s.set_initial(v0, alpha0, beta0)
        s.solve()
        assert np.array_equal(s.get_value(), v)
