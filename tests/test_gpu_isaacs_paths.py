"""The Isaacs kernels at the edges of their dispatch: grids around the sizes
where the wide finest-level phases, the cell-plane tail and the one-block launch
begin, sweep counts without pre- or post-smoothing, capped launches; and the
policy improvement where its float32 screen is least conclusive.

Linear solves are compared with the oracle's direct solve to a tenth of the
path's value bar (as test_policy_solve_parity); improvements with the oracle's
float64 rows: every decision whose gap exceeds 1e-12, ten times the keep-current
tolerance, is the oracle's.
"""
import numpy as np
import pytest

import oracle
from oracle.isaacs import isaacs_game
from test_gpu_isaacs import TOL, rel_err

pytestmark = pytest.mark.gpu

_SYSTEMS = {}


def system(side, variant):
    key = (side, variant)
    if key not in _SYSTEMS:
        game = isaacs_game(side, variant, seed=3)
        rng = np.random.default_rng(11 * side + variant)
        m1 = 5 if variant else 4
        alpha = rng.integers(0, m1, size=game.n).astype(np.uint8)
        beta = rng.integers(0, 4, size=(game.n, m1)).astype(np.uint8)
        _SYSTEMS[key] = (alpha, beta, oracle.solve_policy_system(*oracle.policy_system(game, alpha, beta)))
    return _SYSTEMS[key]


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("sweeps", [(1, 1, -1, -1), (0, 2, 0, 2), (2, 0, 1, 1), (1, 2, 0, 1), (2, 1, 2, 2)])
@pytest.mark.parametrize("side,variant", [(3, 0), (7, 0), (7, 1), (15, 1), (31, 0), (63, 1), (127, 0)])
def test_policy_solve_sweeps(gs, side, variant, sweeps, prec):
    alpha, beta, ref = system(side, variant)
    nu1, nu2, c1, c2 = sweeps
    with gs.GameSolver(precision=prec, nu1=nu1, nu2=nu2, nu1_coarse=c1, nu2_coarse=c2) as s:
        s.set_isaacs_grid(side, variant, 3)
        w, st = s.policy_solve(alpha, beta)
    assert rel_err(w, ref) <= TOL[prec] / 10, st


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("blocks", [1, 2, 7])
@pytest.mark.parametrize("tail_side", [3, 15, 31, 63])
@pytest.mark.parametrize("coarse_max", [1, 9, 49])
def test_policy_solve_launch_shapes(gs, coarse_max, tail_side, blocks, prec):
    alpha, beta, ref = system(127, 0)
    with gs.GameSolver(precision=prec, grid_blocks=blocks, tail_side=tail_side, coarse_max=coarse_max) as s:
        s.set_isaacs_grid(127, 0, 3)
        w, st = s.policy_solve(alpha, beta)
    assert rel_err(w, ref) <= TOL[prec] / 10, st


def smooth_value(side, rng):
    x = np.arange(1, side + 1) / (side + 1)
    v = 0.1 * np.outer(np.sin(np.pi * x), np.sin(np.pi * x))
    for _ in range(3):
        k, l = rng.integers(1, 4, 2)
        v += 0.02 * rng.random() * np.outer(np.sin(k * np.pi * x), np.sin(l * np.pi * x))
    return v.reshape(-1)


def contact_value(game, side, rng):
    """A value touching the obstacle on about half the grid."""
    x = np.arange(1, side + 1) / (side + 1) - 0.5
    psi = (0.2 - (x[:, None] ** 2 + x[None, :] ** 2)).reshape(-1)
    return np.maximum(psi, smooth_value(side, rng))


@pytest.mark.parametrize("kind", ["smooth", "contact", "flat", "large"])
@pytest.mark.parametrize("side,variant", [(1, 0), (1, 1), (3, 1), (31, 0), (63, 1), (127, 0), (255, 1)])
def test_improve_decisions(gs, side, variant, kind):
    import torch
    game = isaacs_game(side, variant, seed=5)
    rng = np.random.default_rng(side)
    m1 = 5 if variant else 4
    v = {"smooth": lambda: smooth_value(side, rng), "contact": lambda: contact_value(game, side, rng),
         "flat": lambda: np.zeros(side * side), "large": lambda: 1e3 * smooth_value(side, rng)}[kind]()
    alpha0 = rng.integers(0, m1, size=game.n).astype(np.uint8)
    beta0 = rng.integers(0, 4, size=(game.n, m1)).astype(np.uint8)
    a_ref, b_ref, fv_ref = oracle.improve(game, v, alpha0, beta0)
    q = oracle.shapley_q(game, v)[:, :m1]
    scale = max(1.0, np.max(np.abs(v)))
    with gs.GameSolver() as s:
        s.set_isaacs_grid(side, variant, 5)
        s.set_initial(alpha0=alpha0, beta0=beta0)
        a, b, fv = s.improve(v)
        # the same through device arrays, and with the result laid over the input
        vd = torch.from_numpy(v).cuda()
        ad = torch.zeros(game.n, dtype=torch.uint8, device="cuda")
        bd = torch.zeros(game.n, m1, dtype=torch.uint8, device="cuda")
        fd = torch.zeros_like(vd)
        for out in (fd, vd):
            st = gs.gamesolve_improve(s.h, vd.data_ptr(), ad.data_ptr(), bd.data_ptr(), out.data_ptr())
            assert st == gs.GS_OK
            assert np.array_equal(ad.cpu().numpy(), a) and np.array_equal(bd.cpu().numpy(), b)
            assert np.array_equal(out.cpu().numpy(), fv)
    assert np.max(np.abs(fv - fv_ref)) <= 1e-14 * scale
    fa = q.min(axis=2)
    srt = np.sort(fa, axis=1)
    sure_a = srt[:, -1] - srt[:, -2] > 1e-12 * scale
    assert np.array_equal(a[sure_a], a_ref[sure_a])
    moves = q[:, :4]
    sb = np.sort(moves, axis=2)
    sure_b = sb[:, :, 1] - sb[:, :, 0] > 1e-12 * scale
    assert np.array_equal(b[:, :4][sure_b], b_ref[:, :4][sure_b])
