"""The finite-game kernels at the edges of their dispatch, against the float64 oracle:
action counts whose rows fill a group of lanes or do not, row lengths with and
without the wide loads, games around the one-block / whole-grid threshold and
around the size below which a game alone must give a batch's bits.

Bars as in test_gpu_games: value 1e-10 relative (float64) / 1e-9 (mixed),
policies bit-exact wherever the oracle's max-min gap exceeds 1e-8.
"""
import numpy as np
import pytest

import synth
from test_gpu_games import TOL, batch, check, oracle_of

pytestmark = pytest.mark.gpu


def solve(gs, n, m1, m2, table, prec, **opts):
    rp, col, prob, rew, mu = table
    with gs.GameSolver(precision=prec, **opts) as s:
        s.set_game(n, m1, m2, rp, col, prob, rew, mu)
        st = s.solve()
        return (s.get_value(), *s.get_policy(), st)


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("m1,m2,k", [(4, 4, 8), (1, 1, 8), (8, 4, 8), (1, 32, 8), (2, 16, 8), (4, 1, 8),
                                     (3, 4, 8), (4, 3, 8), (8, 8, 8), (16, 2, 8), (4, 4, 7), (2, 2, 1), (3, 5, 3)])
@pytest.mark.parametrize("n", [33, 700])
def test_action_counts_and_row_lengths(gs, n, m1, m2, k, prec):
    table = synth.random_game(n, 11 * n + 7 * m1 + m2, m1=m1, m2=m2, k=k, mu=0.95)
    _, ref = oracle_of(n, m1, m2, *table)
    if k == 1:
        # one successor per row: the relaxation does not damp the cycles of such a
        # map, and the evaluation ends at its cycle cap
        with pytest.raises(gs.GameSolveError) as e:
            solve(gs, n, m1, m2, table, prec)
        assert e.value.status == gs.GS_ENOTCONV
        return
    v, a, b, st = solve(gs, n, m1, m2, table, prec)
    assert st["converged"] == 1
    assert check(v, a, b, ref) <= TOL[prec], st


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n", [1100, 40])
def test_rows_of_unequal_length(gs, n, prec):
    """Some successors dropped: substochastic rows of unequal length (read in place)."""
    rp, col, prob, rew, mu = synth.random_game(n, 5 + n, mu=0.95)
    keep = np.ones(len(col), bool)
    keep[np.random.default_rng(n).choice(len(col), len(col) // 9, replace=False)] = False
    lens = np.add.reduceat(keep, rp[:-1])
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    table = (rp, col[keep], prob[keep], rew, mu)
    _, ref = oracle_of(n, 4, 4, *table)
    v, a, b, st = solve(gs, n, 4, 4, table, prec)
    assert st["converged"] == 1
    assert check(v, a, b, ref) <= TOL[prec], st


@pytest.mark.parametrize("prec", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("nu1,nu2", [(1, 1), (2, 1), (0, 1)])
def test_alone_equals_batch_bits(gs, prec, nu1, nu2):
    """Below 4096 states a game gives the same bits alone (one block or the
    whole grid, capped or not) and in a batch."""
    sizes = np.array([31, 511, 512, 513, 1025, 4095])
    (off, rp, col, prob, rew, mu), parts = batch(sizes, 21)
    with gs.GameSolver(precision=prec, nu1=nu1, nu2=nu2) as s:
        s.set_game_batch(off, 4, 4, rp, col, prob, rew, mu)
        assert s.solve()["converged"] == 1
        v = s.get_value()
        a, b = s.get_policy()
    for g, n in enumerate(sizes):
        x0, x1 = off[g], off[g + 1]
        for cap in (0, 5):
            w, c, d, _ = solve(gs, int(n), 4, 4, parts[g], prec, nu1=nu1, nu2=nu2, grid_blocks=cap)
            assert np.array_equal(w, v[x0:x1]) and np.array_equal(c, a[x0:x1]) and np.array_equal(d, b[x0:x1]), (n, cap)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_largest_one_block_games(gs, prec):
    """Sizes whose iterate no longer fits shared memory beside the correction."""
    sizes = np.array([8192, 7300, 300] if prec == "fp64" else [16384, 9000, 300])
    (off, rp, col, prob, rew, mu), parts = batch(sizes, 22)
    with gs.GameSolver(precision=prec) as s:
        s.set_game_batch(off, 4, 4, rp, col, prob, rew, mu)
        assert s.solve()["converged"] == 1
        v = s.get_value()
        a, b = s.get_policy()
    for g, n in enumerate(sizes):
        x0, x1 = off[g], off[g + 1]
        _, ref = oracle_of(int(n), 4, 4, *parts[g])
        assert check(v[x0:x1], a[x0:x1], b[x0:x1], ref) <= TOL[prec], n
