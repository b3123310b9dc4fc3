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
