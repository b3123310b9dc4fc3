"""Isaacs grids where a launch's shape or a solver's history could change a
result: grids of side 31 and below whose coarse levels are not all taken by one
thread block (small tail_side), and calls on a solver after one that met
values that are not finite.

Linear solves are compared with the oracle's direct solve to a tenth of the
path's value bar (as test_policy_solve_parity), whole solves to the bar.
"""
import numpy as np
import pytest

from test_gpu_isaacs import TOL, oracle_solve, rel_err
from test_gpu_isaacs_paths import system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("sweeps", [(1, 1, -1, -1), (1, 2, 0, 1), (0, 2, 0, 2)])
@pytest.mark.parametrize("tail_side", [1, 3, 7, 15])
@pytest.mark.parametrize("side,variant", [(7, 0), (15, 1), (31, 0)])
def test_small_grids_with_grid_wide_coarse_levels(gs, side, variant, tail_side, sweeps, prec):
    alpha, beta, ref = system(side, variant)
    nu1, nu2, c1, c2 = sweeps
    with gs.GameSolver(precision=prec, tail_side=tail_side, nu1=nu1, nu2=nu2, nu1_coarse=c1, nu2_coarse=c2,
                       coarse_max=1) as s:
        s.set_isaacs_grid(side, variant, 3)
        w, st = s.policy_solve(alpha, beta)
    assert rel_err(w, ref) <= TOL[prec] / 10, st


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("tail_side", [3, 7])
def test_fmg_through_small_grids_with_small_tail(gs, tail_side, prec):
    _, ref = oracle_solve(63, 0, 7)
    with gs.GameSolver(precision=prec, tail_side=tail_side, fmg=1, fmg_side=15) as s:
        s.set_isaacs_grid(63, 0, 7)
        st = s.solve()
        v = s.get_value()
    assert st["converged"] == 1 and rel_err(v, ref.v) <= TOL[prec], st


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e300])
@pytest.mark.parametrize("side,variant", [(7, 0), (31, 1), (63, 0), (127, 0)])
def test_good_call_after_one_that_was_not_finite(gs, side, variant, bad, prec):
    """1e300 is finite, but its residual is not in float32."""
    alpha, beta, ref = system(side, variant)
    start = np.zeros(side * side)
    start[[0, side - 1, side * side // 2, side * side - 1]] = bad
    with gs.GameSolver(precision=prec, max_cycles=40) as s:
        s.set_isaacs_grid(side, variant, 3)
        w0, _ = s.policy_solve(alpha, beta)
        s.policy_solve(alpha, beta, w0=start, allow_notconv=True)
        w1, st = s.policy_solve(alpha, beta)
        s.set_initial(v0=start)
        s.solve(allow_notconv=True)
        w2, _ = s.policy_solve(alpha, beta)
    assert np.array_equal(w1, w0) and np.array_equal(w2, w0), st
    assert rel_err(w0, ref) <= TOL[prec] / 10


@pytest.mark.parametrize("side", [8191, 16383])
def test_largest_grids_mixed_against_float64(gs, side):
    """Sides whose rows fill the finest level's staging, and the largest accepted."""
    import ctypes
    import torch
    n = side * side
    gen = torch.Generator(device="cuda").manual_seed(3)
    alpha = torch.randint(0, 4, (n,), dtype=torch.uint8, device="cuda", generator=gen)
    beta = torch.randint(0, 4, (n, 4), dtype=torch.uint8, device="cuda", generator=gen)
    w = {}
    for prec in ("fp64", "mixed", "mixed_bf16"):
        w[prec] = torch.empty(n, dtype=torch.float64, device="cuda")
        with gs.GameSolver(precision=prec, nu2=2) as s:
            s.set_isaacs_grid(side, 0, 1)
            st = gs.gs_solve_stats()
            code = gs.gamesolve_policy_solve(s.h, alpha.data_ptr(), beta.data_ptr(), None, w[prec].data_ptr(),
                                             ctypes.byref(st))
        assert code == gs.GS_OK and st.converged == 1
    scale = float(w["fp64"].abs().max())
    for prec in ("mixed", "mixed_bf16"):
        assert float((w[prec] - w["fp64"]).abs().max()) <= TOL[prec] * scale, prec
