"""Finite games below 4096 states with the block shape chosen by the caller: the
same bits alone and in a batch, on a solver and on a server whatever waits
together."""
import numpy as np
import pytest

import synth
from test_gpu_games import batch
from test_gpu_game_paths import solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("threads", [256, 512])
def test_alone_equals_batch_bits_by_shape(gs, threads, prec):
    sizes = np.array([31, 511, 512, 513, 1025, 3001, 4095])
    (off, rp, col, prob, rew, mu), parts = batch(sizes, 23)
    with gs.GameSolver(precision=prec, game_threads=threads) as s:
        s.set_game_batch(off, 4, 4, rp, col, prob, rew, mu)
        assert s.solve()["converged"] == 1
        v = s.get_value()
        a, b = s.get_policy()
    for g, n in enumerate(sizes):
        x0, x1 = off[g], off[g + 1]
        w, c, d, _ = solve(gs, int(n), 4, 4, parts[g], prec, game_threads=threads)
        assert np.array_equal(w, v[x0:x1]) and np.array_equal(c, a[x0:x1]) and np.array_equal(d, b[x0:x1]), n


@pytest.mark.parametrize("threads", [0, 256, 512])
def test_server_results_do_not_depend_on_the_queue(gs, threads):
    sizes = [600, 3001, 900, 4095, 513]
    tables = [synth.random_game(n, 60 + n) for n in sizes]
    alone = [solve(gs, n, 4, 4, t, "mixed", game_threads=threads)[0] for n, t in zip(sizes, tables)]
    with gs.GameServer(slots=1, precision="mixed", game_threads=threads) as srv:
        # the first request occupies the slot while the others queue up
        tickets = [srv.submit_isaacs(255, 0, 1)] + [srv.submit_game(n, 4, 4, *t) for n, t in zip(sizes, tables)]
        got = [srv.result(t)[0] for t in tickets if srv.wait(t)]
    for n, v, w in zip(sizes, got[1:], alone):
        assert np.array_equal(v, w), n


@pytest.mark.parametrize("threads", [0, 256, 512])
@pytest.mark.parametrize("n", [300, 512, 4095, 4096])
def test_reported_shape_of_a_single_game(gs, n, threads):
    with gs.GameSolver(precision="mixed", game_threads=threads) as s:
        s.set_random_game(n, 4, 4, 3, 0.95)
        s.solve()
        assert s.batch_shape() == (0 if n >= 4096 else threads or 512)


@pytest.mark.parametrize("slots", [2, 4])
def test_large_game_on_a_server_takes_twice_a_slots_share(gs, slots):
    """The blocks of its launch (which the last bits of float64 sums tell apart) do not
    depend on what else is in flight, and on two slots are the whole GPU."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 60_000

    def alone(blocks):
        with gs.GameSolver(precision="fp64", grid_blocks=blocks) as s:
            s.set_random_game(n, 4, 4, 9, 0.99)
            s.solve()
            return s.get_value()

    want = alone(2 * (sms // slots))
    assert not np.array_equal(want, alone(sms // slots))
    with gs.GameServer(slots=slots, precision="fp64") as srv:
        for others in (0, 3):
            t = srv.submit_random_game(n, 4, 4, 9, 0.99)
            rest = [srv.submit_isaacs(255, 0, k + 1) for k in range(others)]
            srv.wait(t)
            v = srv.result(t)[0]
            assert np.array_equal(v, want), others
            for r in rest:
                srv.wait(r)
                srv.result(r)
