"""Timed workloads of the solver, through its public entry points.

A case is one call sequence of a program that uses the library: a whole solve
(new problem data in, value function and policies out) or one layer of the
method that has an entry point of its own (one policy improvement, one
policy-fixed linear solve).  The sizes are those of the library's benchmark
configurations: Isaacs grids of 63^2 to 2047^2 states, random finite games of
1e3 to 1e6 states with 4 x 4 actions and 8 successors, batches of games of 256
to 8192 states, tables of grid games on the algebraic multigrid path, and a mix
of such requests through the server.

Every pass takes the problem data it is given (reward noise, transition tables,
on the device) through set-up, solve and read-out, as a program with a new
problem in hand does.
"""
import ctypes

import numpy as np
import torch

import paper_1107_1653_gb300 as gs

MU = 0.99          # discount of the random finite games
NOISE = 0.05       # half-width of the Isaacs reward noise
SUCC = 8           # successors of a row of a random game


def listed():
    return [
        # A small grid in float64, values and policies: bound by latency,
        # launches and host round trips (the first benchmark configuration).
        {"name": "isaacs_63_fp64", "kind": "isaacs", "side": 63, "variant": 0, "precision": "fp64",
         "nu2": 1, "fmg": False, "noise": NOISE},
        # The headline: one 1023^2 Isaacs solve, float32 cycles in float64 refinement.
        {"name": "isaacs_1023_mixed", "kind": "isaacs", "side": 1023, "variant": 0,
         "precision": "mixed", "nu2": 2, "fmg": False, "noise": NOISE},
        # The same in float64 throughout.
        {"name": "isaacs_1023_fp64", "kind": "isaacs", "side": 1023, "variant": 0,
         "precision": "fp64", "nu2": 2, "fmg": False, "noise": NOISE},
        # The precision configuration: 4.2M states, past the L2.
        {"name": "isaacs_2047_mixed", "kind": "isaacs", "side": 2047, "variant": 0,
         "precision": "mixed", "nu2": 2, "fmg": False, "noise": NOISE},
        # The obstacle game by full multilevel policy iteration from 31^2.
        {"name": "famg_1023_obstacle", "kind": "isaacs", "side": 1023, "variant": 1,
         "precision": "mixed", "nu2": 2, "fmg": True, "noise": NOISE},
        # One policy-fixed linear system (policy evaluation alone) with the
        # coarse operators and weights stored in bfloat16.
        {"name": "policy_solve_511_bf16", "kind": "policy_solve", "side": 511, "variant": 0,
         "precision": "mixed_bf16", "noise": NOISE},
        # One max-min improvement of every state of the obstacle game.
        {"name": "improve_1023_obstacle", "kind": "improve", "side": 1023, "variant": 1,
         "noise": NOISE},
        # A small random game alone (one thread block), float64.
        {"name": "game_3k_fp64", "kind": "game", "n": 3001, "precision": "fp64"},
        # A large random game alone: the whole GPU on one game.
        {"name": "game_500k_mixed", "kind": "game", "n": 500_009, "precision": "mixed"},
        # Many games of unequal size in one call.
        {"name": "batch_1024_mixed", "kind": "batch", "count": 1024, "nmin": 256, "nmax": 8192,
         "precision": "mixed"},
        # A grid game given as explicit transition tables: algebraic multigrid.
        {"name": "tables_127_amg", "kind": "tables", "side": 127, "precision": "mixed", "noise": NOISE},
        # A burst of requests through the server: grids and games of mixed sizes.
        {"name": "serving_20", "kind": "serving", "requests": 20, "slots": 2, "nmax": 300_000,
         "max_side": 1023, "mix": 7},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["isaacs", "isaacs", "famg", "policy_solve", "improve", "game", "game", "batch",
                       "tables", "serving"])
    prec = rng.choice(["fp64", "mixed", "mixed_bf16"])
    noise = round(rng.uniform(0.01, 0.1), 4)
    if kind == "isaacs":
        return {"kind": "isaacs", "side": rng.choice([31, 63, 127, 255, 511, 1023]), "variant": 0,
                "precision": prec, "nu2": rng.choice([1, 2]), "fmg": False, "noise": noise}
    if kind == "famg":
        return {"kind": "isaacs", "side": rng.choice([63, 127, 255, 511]), "variant": rng.choice([0, 1]),
                "precision": prec, "nu2": rng.choice([1, 2]), "fmg": True, "noise": noise}
    if kind == "policy_solve":
        return {"kind": "policy_solve", "side": rng.choice([63, 127, 255, 511, 1023]),
                "variant": rng.choice([0, 1]), "precision": prec, "noise": noise}
    if kind == "improve":
        return {"kind": "improve", "side": rng.choice([63, 127, 255, 511, 1023, 2047]),
                "variant": rng.choice([0, 1]), "noise": noise}
    if kind == "game":
        return {"kind": "game", "n": _log_int(rng, 1000, 500_000), "precision": prec}
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 16, 600), "nmin": _log_int(rng, 64, 512),
                "nmax": _log_int(rng, 1024, 8192), "precision": prec}
    if kind == "tables":
        return {"kind": "tables", "side": rng.randrange(24, 128), "precision": rng.choice(["fp64", "mixed"]),
                "noise": noise}
    return {"kind": "serving", "requests": rng.randrange(6, 17), "slots": rng.choice([1, 2, 4]),
            "nmax": _log_int(rng, 3000, 200_000), "max_side": rng.choice([255, 511, 1023]),
            "mix": rng.randrange(1000)}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _noise(side, half_width, gen):
    u = torch.rand(side * side, dtype=torch.float64, device="cuda", generator=gen)
    return (2.0 * u - 1.0) * half_width


def _random_table(n, gen, rows=None):
    """(row_ptr, col, prob, reward): 4 x 4 actions, SUCC distinct successors per
    row in increasing order, Dirichlet(1) probabilities, rewards U(-1, 1)."""
    rows = n * 16 if rows is None else rows
    col = torch.rand(rows, SUCC, dtype=torch.float64, device="cuda", generator=gen)
    col = (col * (n - SUCC + 1)).long().clamp_(max=n - SUCC).sort(dim=1).values
    col = (col + torch.arange(SUCC, device="cuda")).to(torch.int32)
    p = -torch.log1p(-torch.rand(rows, SUCC, dtype=torch.float64, device="cuda", generator=gen))
    p /= p.sum(dim=1, keepdim=True)
    rew = 2.0 * torch.rand(rows, dtype=torch.float64, device="cuda", generator=gen) - 1.0
    row_ptr = torch.arange(rows + 1, dtype=torch.int64, device="cuda") * SUCC
    return row_ptr, col.reshape(-1), p.reshape(-1), rew


def _batch_table(case, gen, sizes):
    """Tables of the batch's games one after the other (columns within a game)."""
    parts = [_random_table(int(n), gen)[1:] for n in sizes]
    col, prob, rew = (torch.cat([p[k] for p in parts]) for k in range(3))
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64))
    row_ptr = torch.arange(rew.numel() + 1, dtype=torch.int64, device="cuda") * SUCC
    return off, row_ptr, col, prob, rew


STEPS = ((1, 0), (-1, 0), (0, 1), (0, -1))   # actions +x1, -x1, +x2, -x2


def _isaacs_consts(side):
    h = 1.0 / (side + 1)
    return h, 2.0 + h, 1.0 / (1.0 + h * h), h * h / (1.0 + h * h)


def _isaacs_rows(side, xi):
    """The Isaacs game's rows: probabilities [4, 4, 5] towards E, W, N, S and the
    state itself, and rewards [4, 4, n]."""
    h, c0, _, kappa = _isaacs_consts(side)
    p = torch.zeros(4, 4, 5, dtype=torch.float64, device="cuda")
    for a in range(4):
        for b in range(4):
            for d in range(4):
                drift = 0.5 * sum((STEPS[a][k] - STEPS[b][k]) * STEPS[d][k] for k in range(2))
                p[a, b, d] = (0.5 + h * max(drift, 0.0)) / c0
            p[a, b, 4] = h / c0 if a == b else 0.0
    x = torch.arange(1, side + 1, dtype=torch.float64, device="cuda") * h
    s = torch.sin(torch.pi * x)
    base = (s[:, None] * s[None, :]).reshape(-1) + xi
    ab = torch.arange(4, dtype=torch.float64, device="cuda")
    r = kappa * (base[None, None, :] + 0.1 * (ab[:, None] - ab[None, :])[:, :, None])
    return p, r


def _obstacle(side):
    x = torch.arange(1, side + 1, dtype=torch.float64, device="cuda") / (side + 1) - 0.5
    return (0.2 - (x[:, None] ** 2 + x[None, :] ** 2)).reshape(-1)


def _neighbours(v, side):
    g = torch.nn.functional.pad(v.reshape(side, side), (1, 1, 1, 1))
    return torch.stack([g[1:-1, 2:], g[1:-1, :-2], g[2:, 1:-1], g[:-2, 1:-1], g[1:-1, 1:-1]]).reshape(5, -1)


def _isaacs_values(v, side, variant, xi):
    """F(v; x, a, b) minimised over b for every a [m1, n], and the minimisers."""
    p, r = _isaacs_rows(side, xi)
    mu = _isaacs_consts(side)[2]
    nb = _neighbours(v, side)
    best, reply = [], []
    for a in range(4):
        m = (mu * (p[a] @ nb) + r[a]).min(dim=0)
        best.append(m.values)
        reply.append(m.indices)
    if variant == 1:
        best.append(_obstacle(side))
        reply.append(torch.zeros_like(reply[0]))
    return torch.stack(best), torch.stack(reply)


def _greedy(v, side, variant, xi):
    best, reply = _isaacs_values(v, side, variant, xi)
    alpha = best.max(dim=0).indices
    return alpha.to(torch.uint8), reply.t().contiguous().to(torch.uint8)


def _guess(side, gen):
    """A value function as policy iteration meets it: smooth, with the game's size."""
    x = torch.arange(1, side + 1, dtype=torch.float64, device="cuda") / (side + 1)
    s, t = torch.sin(torch.pi * x), torch.sin(2 * torch.pi * x)
    w = torch.rand(4, dtype=torch.float64, device="cuda", generator=gen) * 0.02
    v = 0.1 * s[:, None] * s[None, :] + w[0] * t[:, None] * s[None, :] + w[1] * s[:, None] * t[None, :]
    return (v + w[2] * t[:, None] * t[None, :]).reshape(-1).contiguous()


def _grid_tables(side, xi):
    """The Isaacs game as transition tables in CSR form (neighbours on the
    boundary dropped)."""
    n = side * side
    p, r = _isaacs_rows(side, xi)
    x = torch.arange(n, device="cuda")
    i, j = x % side, x // side
    inside = torch.stack([i + 1 < side, i > 0, j + 1 < side, j > 0, torch.ones_like(i, dtype=torch.bool)])
    target = torch.stack([x + 1, x - 1, x + side, x - side, x])
    on = inside.t()[:, None, None, :] & (p > 0)[None]          # [n, 4, 4, 5]
    col = target.t()[:, None, None, :].expand(n, 4, 4, 5)[on].to(torch.int32)
    prob = p[None].expand(n, 4, 4, 5)[on]
    row_ptr = torch.zeros(n * 16 + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = on.sum(dim=3).reshape(-1).cumsum(0)
    reward = r.permute(2, 0, 1).reshape(-1).contiguous()
    return row_ptr, col, prob.contiguous(), reward


def _sizes(case, seed):
    """Batch: sizes U{nmin .. nmax} (one list per seed, the same total to within a few states)."""
    u = (np.arange(case["count"]) + 0.5) / case["count"]
    sizes = case["nmin"] + np.floor(u * (case["nmax"] - case["nmin"] + 1)).astype(np.int64)
    return np.random.RandomState(seed % (1 << 31)).permutation(sizes)


def _requests(case):
    """Serving mix: 70% Isaacs grids, 30% random games of log-uniform size,
    in an order fixed by the case."""
    rs = np.random.RandomState(case["mix"])
    sides = [s for s in (63, 127, 255, 511, 1023) if s <= case["max_side"]]
    out = []
    for k in range(case["requests"]):
        if k % 10 in (2, 5, 8):
            out.append(("game", int(round(1000 * (case["nmax"] / 1000) ** rs.rand()))))
        else:
            out.append(("isaacs", int(sides[rs.randint(len(sides))])))
    return [out[k] for k in rs.permutation(len(out))]


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    st = {"case": case}
    stream = torch.cuda.current_stream()
    if kind == "serving":
        st["server"] = gs.GameServer(slots=case["slots"], precision="mixed", nu1=1, nu2=2)
        rs = np.random.RandomState(seed % (1 << 31))
        st["requests"] = []
        for what, size in _requests(case):
            if what == "game":
                st["requests"].append((what, size, _random_table(size, gen)))
            else:
                st["requests"].append((what, size, int(rs.randint(1, 1 << 30))))
        torch.cuda.synchronize()   # the server's workers read the tables on streams of their own
        return st
    if kind in ("isaacs", "policy_solve", "improve"):
        side, variant = case["side"], case["variant"]
        n, m1 = side * side, 5 if variant == 1 else 4
        st["xi"] = _noise(side, case["noise"], gen)
        opts = {"precision": case.get("precision", "fp64"), "stream": stream, "nu1": 1, "nu2": case.get("nu2", 2)}
        if case.get("fmg"):
            opts.update(fmg=1, fmg_side=31, fmg_c=0.01 if variant == 1 else 0.1)
        st["solver"] = gs.GameSolver(**opts)
        st["value"] = torch.empty(n, dtype=torch.float64, device="cuda")
        if kind == "isaacs":
            # Policies are part of the result up to 127^2.  On larger grids some of
            # the millions of entries tie within the keep-current tolerance, and which
            # of the tied actions stays depends on the iterates, not on the game.
            if side <= 127:
                st["alpha"] = torch.empty(n, dtype=torch.uint8, device="cuda")
                st["beta"] = torch.empty(n, m1, dtype=torch.uint8, device="cuda")
            return st
        st["solver"].set_isaacs_grid(side, variant, 1, st["xi"])
        st["v0"] = _guess(side, gen)
        alpha, beta = _greedy(st["v0"], side, variant, st["xi"])
        if kind == "policy_solve":
            st["given"] = alpha, beta
        else:
            # improvement: the current policies are those of a slightly different value
            w = _guess(side, gen)
            a0, b0 = _greedy(w, side, variant, st["xi"])
            st["solver"].set_initial(None, a0, b0)
            st["alpha"], st["beta"] = torch.empty_like(alpha), torch.empty_like(beta)
        return st
    if kind == "tables":
        side = case["side"]
        st["n"], st["mu"] = side * side, _isaacs_consts(side)[2]
        st["table"] = _grid_tables(side, _noise(side, case["noise"], gen))
        opts = {"game_solver": 1}
    elif kind == "game":
        st["n"], st["mu"] = case["n"], MU
        st["table"] = _random_table(case["n"], gen)
        opts = {}
    else:
        sizes = _sizes(case, seed)
        st["offsets"], *st["table"] = _batch_table(case, gen, sizes)
        st["mu"] = torch.full((len(sizes),), MU, dtype=torch.float64)
        st["n"] = int(sizes.sum())
        opts = {"game_threads": 512}
    st["solver"] = gs.GameSolver(precision=case["precision"], stream=stream, **opts)
    st["value"] = torch.empty(st["n"], dtype=torch.float64, device="cuda")
    st["alpha"] = torch.empty(st["n"], dtype=torch.uint8, device="cuda")
    st["beta"] = torch.empty(st["n"], 4, dtype=torch.uint8, device="cuda")
    return st


# ------------------------------------------------------------------ one pass
def _ok(status):
    if status != gs.GS_OK:
        raise RuntimeError("status %d: %s" % (status, gs.gamesolve_last_error().decode()))


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "serving":
        srv = st["server"]
        tickets = []
        for what, size, data in st["requests"]:
            if what == "game":
                row_ptr, col, prob, rew = data
                tickets.append(srv.submit_game(size, 4, 4, row_ptr, col, prob, rew, MU, borrow=True))
            else:
                tickets.append(srv.submit_isaacs(size, 0, data))
        for t in tickets:
            srv.wait(t)
        return [srv.result(t)[0] for t in tickets]
    s = st["solver"]
    if kind == "improve":
        a, b, fv = st["alpha"], st["beta"], st["value"]
        _ok(gs.gamesolve_improve(s.h, st["v0"].data_ptr(), a.data_ptr(), b.data_ptr(), fv.data_ptr()))
        return {"alpha": a, "beta": b, "value": fv}
    if kind == "policy_solve":
        alpha, beta = st["given"]
        stats = gs.gs_solve_stats()
        _ok(gs.gamesolve_policy_solve(s.h, alpha.data_ptr(), beta.data_ptr(), st["v0"].data_ptr(),
                                      st["value"].data_ptr(), ctypes.byref(stats)))
        return {"value": st["value"]}
    if kind == "isaacs":
        s.set_isaacs_grid(case["side"], case["variant"], 1, st["xi"])
    elif kind == "batch":
        s.set_game_batch(st["offsets"], 4, 4, *st["table"], st["mu"])
    else:
        s.set_game(st["n"], 4, 4, *st["table"], st["mu"])
    s.solve()
    out = {"value": s.get_value(st["value"])}
    if "alpha" in st:
        out["alpha"], out["beta"] = s.get_policy(st["alpha"], st["beta"])
    return out


# ------------------------------------------------------------------ work
def _grid_work(n, noise_in):
    # noise in (grids given as tensors), value out; one evaluation of the
    # policy-fixed rows and one improvement of every state
    return (16 if noise_in else 8) * n, (10 + 16 * 12) * n


def _table_work(n):
    # row pointers, columns, probabilities and rewards in; value and policies
    # out; one evaluation of all rows
    return 16 * n * (8 + 12 * SUCC + 8) + 13 * n, 16 * n * (2 * SUCC + 3)


def work(case):
    kind = case["kind"]
    if kind == "serving":
        parts = [_table_work(size) if what == "game" else _grid_work(size * size, False)
                 for what, size in _requests(case)]
        nbytes, flops = (sum(p[k] for p in parts) for k in range(2))
    elif kind == "batch":
        nbytes, flops = _table_work(int(_sizes(case, 0).sum()))
    elif kind == "game":
        nbytes, flops = _table_work(case["n"])
    elif kind == "tables":
        n = case["side"] ** 2
        nbytes, flops = 16 * n * (8 + 12 * 4 + 8) + 13 * n, 16 * n * 11
    elif kind == "improve":
        n = case["side"] ** 2
        m1 = 5 if case["variant"] == 1 else 4
        nbytes, flops = n * (8 + 8 + 2 * (1 + m1) + 8), 16 * 12 * n   # v, rewards, policies in and out, F(v)
    elif kind == "policy_solve":
        n = case["side"] ** 2
        m1 = 5 if case["variant"] == 1 else 4
        nbytes, flops = n * (1 + m1 + 8 + 8 + 8), 10 * n              # policies, rewards, guess in; value out
    else:
        nbytes, flops = _grid_work(case["side"] ** 2, True)
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ 64-bit values
def _grid_system(side, variant, xi, alpha, beta):
    """Row entries [5, n] of I - mu P (E, W, N, S, diagonal) and the right-hand
    side of the system fixed by alpha [n] and beta [n, m1]."""
    p, r = _isaacs_rows(side, xi)
    mu = _isaacs_consts(side)[2]
    n = side * side
    a = alpha.long()
    b = beta.long().gather(1, a[:, None])[:, 0]
    stop = a == 4
    ai = torch.where(stop, torch.zeros_like(a), a)
    row = -mu * p[ai, b].t().contiguous()
    row[4] += 1.0
    rhs = r[ai, b, torch.arange(n, device="cuda")]
    if variant == 1:
        row[:4, stop] = 0.0
        row[4, stop] = 1.0
        rhs = torch.where(stop, _obstacle(side), rhs)
    return row, rhs


def _grid_solve(side, row, rhs):
    """Block tridiagonal elimination (one block per grid line), refined once."""
    E, W, N, S, D = row.reshape(5, side, side)
    inv = []
    for j in range(side):
        A = torch.diag(D[j]) + torch.diag(E[j, :-1], 1) + torch.diag(W[j, 1:], -1)
        if j:
            A -= S[j][:, None] * inv[-1] * N[j - 1][None, :]
        inv.append(torch.linalg.inv(A))

    def solve(f):
        f = f.reshape(side, side)
        y = []
        for j in range(side):
            y.append(inv[j] @ (f[j] if j == 0 else f[j] - S[j] * y[-1]))
        for j in range(side - 2, -1, -1):
            y[j] = y[j] - inv[j] @ (N[j] * y[j + 1])
        return torch.stack(y).reshape(-1)

    v = solve(rhs)
    for _ in range(2):
        v = v + solve(rhs - (row * _neighbours(v, side)).sum(dim=0))
    return v


def _grid_game(side, variant, xi):
    """Value of the Isaacs game by policy iteration with direct solves."""
    v = torch.zeros(side * side, dtype=torch.float64, device="cuda")
    alpha, beta = _greedy(v, side, variant, xi)
    for _ in range(400):
        for _ in range(100):   # MIN's replies at fixed alpha
            v = _grid_solve(side, *_grid_system(side, variant, xi, alpha, beta))
            best, reply = _isaacs_values(v, side, variant, xi)
            a = alpha.long()[None]
            old = _row_value(side, variant, xi, v, alpha, beta)
            gain = old - best.gather(0, a)[0]
            beta = torch.where((gain > 1e-14)[:, None], reply.t().to(torch.uint8), beta)
            if not bool((gain > 1e-14).any()):
                break
        gain = best.max(dim=0)
        better = gain.values - best.gather(0, alpha.long()[None])[0] > 1e-14
        if not bool(better.any()):
            return v
        alpha = torch.where(better, gain.indices.to(torch.uint8), alpha)
        beta = torch.where(better[:, None], reply.t().to(torch.uint8), beta)
    return v


def _row_value(side, variant, xi, v, alpha, beta):
    row, rhs = _grid_system(side, variant, xi, alpha, beta)
    return rhs + v - (row * _neighbours(v, side)).sum(dim=0)


def _table_game(sizes, table):
    """Values of random games by iterating the Shapley operator, each game's
    iterate shifted by the constant that closes its mean gap."""
    _, col, prob, rew = table
    sizes = torch.as_tensor(np.asarray(sizes), device="cuda")
    count = len(sizes)
    game = torch.repeat_interleave(torch.arange(count, device="cuda"), sizes)
    first = torch.cumsum(sizes, 0) - sizes
    n = len(game)
    v = torch.zeros(n, dtype=torch.float64, device="cuda")
    part = 1 << 18

    def shapley(v):
        f = torch.empty_like(v)
        for lo in range(0, n, part):
            hi = min(n, lo + part)
            c = col[lo * 16 * SUCC:hi * 16 * SUCC].view(hi - lo, 16 * SUCC).long() + first[game[lo:hi]][:, None]
            q = (prob[lo * 16 * SUCC:hi * 16 * SUCC].view(hi - lo, 16, SUCC) *
                 v[c].view(hi - lo, 16, SUCC)).sum(dim=2) * MU + rew[lo * 16:hi * 16].view(hi - lo, 16)
            f[lo:hi] = q.view(hi - lo, 4, 4).min(dim=2).values.max(dim=1).values
        return f

    for _ in range(400):
        f = shapley(v)
        gap = torch.zeros(count, dtype=torch.float64, device="cuda").index_add_(0, game, f - v) / sizes
        step = f + (gap * MU / (1.0 - MU))[game]
        if float((step - v).abs().max()) < 4e-15 * float(step.abs().max()):
            return step
        v = step
    return v


def exact(case, seed):
    """The same results by dense or fixed-point arithmetic in float64.  None
    where that takes too long (policy iteration on the large grids) and for the
    policies, which are whole numbers and compared as they are."""
    kind = case["kind"]
    if kind == "isaacs" and case["side"] > (63 if case["variant"] == 1 else 255):
        return None
    if kind == "serving":
        gen, out = _generator(seed), []
        for what, size in _requests(case):
            out.append(_table_game([size], _random_table(size, gen)) if what == "game" else None)
        return out
    gen = _generator(seed)
    policies = {"alpha": None, "beta": None}
    if kind == "game":
        return {"value": _table_game([case["n"]], _random_table(case["n"], gen)), **policies}
    if kind == "batch":
        sizes = _sizes(case, seed)
        return {"value": _table_game(sizes, _batch_table(case, gen, sizes)[1:]), **policies}
    side, variant = case["side"], case.get("variant", 0)
    xi = _noise(side, case["noise"], gen)
    if kind == "tables":
        return {"value": _grid_game(side, 0, xi), **policies}
    if kind == "isaacs":
        return {"value": _grid_game(side, variant, xi), **(policies if side <= 127 else {})}
    v0 = _guess(side, gen)
    if kind == "improve":
        return {"value": _isaacs_values(v0, side, variant, xi)[0].max(dim=0).values, **policies}
    alpha, beta = _greedy(v0, side, variant, xi)
    return {"value": _grid_solve(side, *_grid_system(side, variant, xi, alpha, beta))}
