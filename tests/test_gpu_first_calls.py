"""Calls on a grid that has just been set, before any solve or start: they use the
default start (v = 0, action 0 or stop everywhere, replies 0), not what the
memory held."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def fill_memory(gs, side, value):
    """Leaves `value` in the device memory a grid of this side is cut from."""
    import ctypes
    import torch
    n = side * side
    a = torch.zeros(n, dtype=torch.uint8, device="cuda")
    b = torch.full((n, 4), 3, dtype=torch.uint8, device="cuda")
    start = torch.full((n,), value, dtype=torch.float64, device="cuda")
    w = torch.empty_like(start)
    with gs.GameSolver(max_cycles=1) as s:
        s.set_isaacs_grid(side, 0, 1)
        gs.gamesolve_policy_solve(s.h, a.data_ptr(), b.data_ptr(), start.data_ptr(), w.data_ptr(), None)


@pytest.mark.parametrize("variant", [0, 1])
@pytest.mark.parametrize("side", [15, 63, 127])
def test_improve_before_any_start(gs, side, variant):
    n, m1 = side * side, 5 if variant else 4
    v = 0.1 * np.random.default_rng(side).uniform(size=n)
    alpha = np.full(n, 4 if variant else 0, np.uint8)
    beta = np.zeros((n, m1), np.uint8)
    given = np.random.default_rng(1).integers(0, m1, n).astype(np.uint8)
    with gs.GameSolver() as s:
        fill_memory(gs, side, np.nan)
        s.set_isaacs_grid(side, variant, 2)
        got = s.improve(v)
        s.set_initial(None, alpha, beta)
        want = s.improve(v)
        s.set_isaacs_grid(side, variant, 2)
        s.set_initial(None, given, None)
        got_alpha = s.improve(v)
        s.set_initial(None, given, beta)
        want_alpha = s.improve(v)
    for x, y in zip(got + got_alpha, want + want_alpha):
        assert np.array_equal(x, y)


def test_full_multilevel_that_stops_on_a_coarse_grid(gs):
    """The finest grid is not reached: its value and policies are the default start."""
    side = 127
    fill_memory(gs, side, np.nan)
    with gs.GameSolver(precision="mixed", max_cycles=1, fmg=1, fmg_side=15) as s:
        s.set_isaacs_grid(side, 1, 1)
        st = s.solve(allow_notconv=True)
        v = s.get_value()
        alpha, beta = s.get_policy()
    assert st["converged"] == 0 and st["fmg_levels"] < 4
    assert not v.any() and np.all(alpha == 4) and not beta.any()
