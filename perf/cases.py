"""The work whose speed is measured: what a program that uses this framework has it do.

Three kinds of users' programs stand behind the cases: one that solves a game
(``cfr.Solver``: iterations from a fresh state, then the strategies; and the
exact best response to a strategy), one that serves many re-solves at once
(the batched launches of a serving round, and ``serve.Server`` as a whole),
and one that trains or applies the warm-start network (``mlp.MLP``). Games
are the repository's own synthetic families at the sizes of its tests and
benchmark: one-card poker, endgames of 1e3 to 1e6 edges, random trees, and
the two-round card game on decks that compile in a few seconds.

A game's structure belongs to the case; the seed draws what changes from one
solve to the next: the ranges (the chance probabilities of the deal at the
root) of the card games and endgames, the payoffs of the random trees, the
strategy that a best response is computed against, the network's weights and
training rows.

``exact`` computes the same results in 64 bits with plain torch operations,
level by level from the tabular game: no code of the solver is used there.
"""
import dataclasses
import functools
import math

import numpy as np
import torch

import gamegen as gg
from paper_2609_11923_gb300 import cfr, mlp, serve, warmstart

# ----------------------------------------------------------------- the cases
# "solve": Solver.reset, iterate(iters), then the average and the current
#   strategy on the device. "tune" as the benchmark does for its large games.
# "evaluate": Solver.best_response() of a given average strategy.
# "round": one round of a static batch of endgames, as the server runs it:
#   `iters` iterations of every game in one launch, one exploitability
#   launch, and the average strategies on the device.
# "serve": Server.serve() of requests that all wait at time 0, host work
#   (compiling the games) included.
# "train", "predict": one step of the warm-start network, one inference.

# Fields of a solve: precision 32 or 64; rule 0 CFR+, 1 CFR, 2 PCFR+; order 0
# simultaneous, 1 alternating.


def listed():
    return [
        # the smallest call there is: one-card poker, 301 nodes (the smoke
        # test's game); one check interval of the stop rule
        {"name": "solve_tiny_p32", "kind": "solve", "game": "tiny", "a": 5, "b": 2, "precision": 32, "rule": 0,
         "order": 0, "iters": 50, "tune": False},
        # a real-time re-solve of one subgame, as serve.solve_alone does it
        {"name": "solve_endgame_p32", "kind": "solve", "game": "endgame", "a": 3, "b": 20000, "precision": 32,
         "rule": 0, "order": 0, "iters": 50, "tune": False},
        # the benchmark's random tree (2.8M nodes, irregular, sets of 1-16)
        {"name": "solve_tree_p32", "kind": "solve", "game": "tree", "a": 0, "b": 14, "precision": 32, "rule": 0,
         "order": 0, "iters": 5, "tune": True},
        # parity mode on an irregular game, with the other update rule and
        # order that convergence studies use
        {"name": "solve_tree_p64", "kind": "solve", "game": "tree", "a": 1, "b": 12, "precision": 64, "rule": 2,
         "order": 1, "iters": 10, "tune": False},
        # the largest: the two-round card game with the benchmark's betting
        # on a 21-card deck (27M nodes, far larger than L2)
        {"name": "solve_card_p32", "kind": "solve", "game": "card", "a": 7, "b": 3, "precision": 32, "rule": 0,
         "order": 0, "iters": 10, "tune": True},
        # the same family in parity mode (18-card deck, 11M nodes)
        {"name": "solve_card_p64", "kind": "solve", "game": "card", "a": 6, "b": 3, "precision": 64, "rule": 0,
         "order": 0, "iters": 5, "tune": True},
        # how far from equilibrium a strategy is: run after every few hundred
        # iterations of a large solve
        {"name": "evaluate_card", "kind": "evaluate", "game": "card", "a": 6, "b": 3, "precision": 32},
        # a serving round: 64 uneven subgames, one CTA each
        {"name": "round_mixed", "kind": "round", "n": 64, "lo": 1000, "hi": 200000, "a": 100, "iters": 50,
         "cluster": 1, "precision": 32},
        # a serving round of the large requests, run as clusters
        {"name": "round_large", "kind": "round", "n": 10, "lo": 200000, "hi": 1000000, "a": 300, "iters": 50,
         "cluster": 8, "precision": 32},
        # the server as a whole, from requests to strategies
        {"name": "serve_mixed", "kind": "serve", "n": 32, "lo": 1000, "hi": 300000, "a": 500, "iters": 50},
        # the warm-start network at warmstart.train's batch size
        {"name": "mlp_train", "kind": "train", "rows": 4096},
        # one inference over every set of a batch of games
        {"name": "mlp_predict", "kind": "predict", "rows": 200000},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def options():
        return {"rule": rng.choice([0, 0, 1, 2]), "order": rng.choice([0, 0, 1]), "tune": rng.random() < 0.5}

    kind = rng.choice(["solve", "solve", "solve", "evaluate", "round", "round", "serve", "train", "predict"])
    if kind in ("solve", "evaluate"):
        game = rng.choice(["tiny", "endgame", "endgame", "tree", "card"])
        c = {"kind": kind, "game": game, "precision": rng.choice([32, 32, 64])}
        if game == "tiny":
            c.update(a=rng.randint(3, 13), b=rng.randint(1, 4))
        elif game == "endgame":
            c.update(a=rng.randint(0, 1 << 20), b=log_int(1000, 1000000))
        elif game == "tree":
            c.update(a=rng.randint(0, 1 << 20), b=rng.randint(5, 13))
        else:
            a, b = rng.choice([(3, 2), (4, 2), (3, 3), (5, 2), (4, 3), (6, 2), (5, 3), (6, 3), (4, 4)])
            c.update(a=a, b=b, stride=rng.randint(1, 9))
        if kind == "solve":
            c.update(options(), iters=rng.randint(3, 6) if game == "tree" else rng.randint(5, 20))
        return c
    if kind == "round":
        big = rng.random() < 0.3
        n = rng.randint(2, 10) if big else log_int(3, 200)
        precision = 32 if big else rng.choice([32, 32, 32, 64])
        lo, hi = (200000, 1000000) if big else (1000, log_int(4000, 200000 if precision == 32 else 25000))
        return {"kind": kind, "n": n, "lo": lo, "hi": hi, "a": rng.randint(0, 1 << 20), "iters": 50,
                "cluster": 8 if big else 1, "precision": precision}
    if kind == "serve":
        return {"kind": kind, "n": log_int(4, 48), "lo": 1000, "hi": log_int(10000, 300000),
                "a": rng.randint(0, 1 << 20), "iters": 50}
    if kind == "train":
        return {"kind": kind, "rows": log_int(256, 8192)}
    return {"kind": kind, "rows": log_int(50, 200000)}


# ----------------------------------------------------------------- the games
@functools.lru_cache(maxsize=16)
def _build(game, a, b, stride):
    if game == "tiny":
        return gg.tiny_card(a, b)
    if game == "endgame":
        return gg.endgame(a, b)
    if game == "tree":
        return gg.random_tree(a, depth=b)
    return gg.large_card(a, b, 2, 3) if stride == 1 else gg.large_card_sampled(stride, a, b, 2, 3)


def _structure(case):
    """Ranks and bets a round (tiny), generator seed and edges (endgame) or
    depth (tree), ranks and suits (card; every stride-th deal)."""
    return _build(case["game"], case["a"], case["b"], case.get("stride", 1))


def _seeded(g, seed):
    """The game with this seed's deal probabilities (a chance root), or
    payoffs (else)."""
    rng = np.random.default_rng(seed)
    if g.kind[0] == gg.CHANCE and int(g.child_begin[1]) >= 6:
        p = g.chance_prob.copy()
        n = int(g.child_begin[1])
        p[:n] *= rng.gamma(2.0, size=n)
        p[:n] /= p[:n].sum()
        return dataclasses.replace(g, chance_prob=p)
    u = np.where(g.kind == gg.TERMINAL, rng.uniform(-1.0, 1.0, g.n_nodes), 0.0)
    return dataclasses.replace(g, payoff=u)


def _game(case, seed):
    return _seeded(_structure(case), seed)


@functools.lru_cache(maxsize=4)
def _sizes(n, lo, hi, a):
    """Edge targets log-uniform in [lo, hi] and generator seeds of a batch."""
    rng = np.random.default_rng(a)
    return [(a + i, int(np.exp(rng.uniform(np.log(lo), np.log(hi))))) for i in range(n)]


@functools.lru_cache(maxsize=4)
def _batch_structures(n, lo, hi, a):
    return [gg.endgame(s, e) for s, e in _sizes(n, lo, hi, a)]


def _batch(case, seed):
    gs = _batch_structures(case["n"], case["lo"], case["hi"], case["a"])
    return [_seeded(g, 1000003 * seed + i) for i, g in enumerate(gs)]


def _some_average(g, seed):
    """A strategy sum as a solve leaves it: every slot positive, uneven."""
    return np.random.default_rng(seed).gamma(0.5, size=g.n_slots) + 1e-6


def _rows(case, seed):
    """Feature rows like warmstart.features': one-hot groups and a few reals."""
    r = torch.Generator(device="cuda").manual_seed(seed)
    B, F = case["rows"], warmstart.F_IN
    X = (torch.rand(B, F, generator=r, device="cuda") < 0.08).float()
    X[:, 168:173] = torch.rand(B, 5, generator=r, device="cuda") * 2.0 - 1.0
    nact = torch.randint(2, mlp.N_OUT + 1, (B,), generator=r, device="cuda", dtype=torch.int32)
    T = torch.rand(B, mlp.N_OUT, generator=r, device="cuda") + 1e-3
    T = T * (torch.arange(mlp.N_OUT, device="cuda") < nact[:, None])
    return X, nact, T / T.sum(1, keepdim=True)


# ------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "evaluate"):
        g = _game(case, seed)
        s = cfr.Solver(g, precision=cfr.P32 if case["precision"] == 32 else cfr.P64, rule=case.get("rule", 0),
                       order=case.get("order", 0))
        if kind == "evaluate":
            avg = _some_average(g, seed)
            s.set_state(np.zeros(g.n_slots), avg, 1)
        elif case["tune"]:
            s.autotune()
        current = torch.empty(s.n_slots, dtype=torch.float64, device="cuda")
        return {"kind": kind, "solver": s, "iters": case.get("iters", 0), "current": current}
    if kind == "round":
        specs = _batch(case, seed)
        opts = cfr.make_options(precision=cfr.P32 if case["precision"] == 32 else cfr.P64)
        hs = warmstart.compile_many(specs, opts)
        sizes = [cfr.cfr_plan(h) for h in hs]
        pool = serve.DevicePool(sum(n + serve.ALIGN for n in sizes) + serve.ALIGN)
        s = int(torch.cuda.current_stream().cuda_stream)
        for h, n in zip(hs, sizes):
            cfr.cfr_bind(h, pool.ptr(pool.alloc(n)), n, s)
        tb = cfr.cfr_batch_table_bytes(len(hs))
        table = torch.empty(tb + 16, dtype=torch.uint8, device="cuda")
        slots = [g.n_slots for g in specs]
        return {"kind": kind, "batch": _Handles(hs), "pool": pool, "table": table, "table_bytes": tb,
                "strategy": torch.empty(sum(slots), dtype=torch.float64, device="cuda"), "slots": slots,
                "iters": case["iters"], "cluster": case["cluster"]}
    if kind == "serve":
        specs = _batch(case, seed)
        # the launch shape that serve.autotune_batch picks for these games
        srv = serve.Server(pool_bytes=1 << 29, max_active=64, threads=1024, lanes=8, check_every=25,
                           max_iters=case["iters"], target=0.0, keep_strategies=True)
        return {"kind": kind, "server": srv, "requests": [serve.Request(i, g) for i, g in enumerate(specs)]}
    X, nact, T = _rows(case, seed)
    return {"kind": kind, "net": _network(seed), "X": X, "nact": nact, "T": T}


STEPS = 100  # training steps behind the network


def _network(seed):
    """A network in the middle of its training: biases and Adam moments too."""
    net = mlp.MLP(warmstart.F_IN, seed=seed % (1 << 31))
    r = torch.Generator(device="cuda").manual_seed(seed + 1)
    like = lambda x: torch.randn(x.shape, generator=r, device="cuda")  # noqa: E731
    for x in net.b:
        x.copy_(0.1 * like(x))
    for m, v in zip(net.mW + net.mb, net.vW + net.vb):
        m.copy_(1e-4 * like(m))
        v.copy_(1e-6 * (0.5 + like(v).square()))
    net.step_no = STEPS
    return net


class _Handles:
    """Compiled games that are released with the state that holds them."""

    def __init__(self, hs):
        self.hs = hs

    def __del__(self):
        for h in self.hs:
            cfr.cfr_destroy(h)


def run(state):
    kind = state["kind"]
    if kind == "solve":
        s = state["solver"]
        s.reset()
        s.iterate(state["iters"])
        cfr.cfr_current_strategy(s.h, state["current"].data_ptr(), True, s._s())
        return {"average": s.avg_strategy_device(), "current": state["current"]}
    if kind == "evaluate":
        return list(state["solver"].best_response())
    if kind == "round":
        hs, s = state["batch"].hs, int(torch.cuda.current_stream().cuda_stream)
        tp = (state["table"].data_ptr() + 15) & ~15
        cfr.cfr_batch_iterate(hs, state["iters"], tp, state["table_bytes"], 1024, 8, s, cluster=state["cluster"])
        ex = cfr.cfr_batch_exploitability(hs, tp, state["table_bytes"], 1024, 8, s)
        out, at = state["strategy"], 0
        for h, n in zip(hs, state["slots"]):
            cfr.cfr_avg_strategy(h, out[at:].data_ptr(), True, s)
            at += n
        return {"exploitability": ex, "average": out}
    if kind == "serve":
        got = sorted(state["server"].serve(state["requests"]), key=lambda r: r.rid)
        return {"exploitability": np.array([r.exploitability for r in got]),
                "iterations": np.array([r.iterations for r in got]),
                "average": np.concatenate([r.strategy for r in got])}
    net = state["net"]
    if kind == "train":
        loss = net.loss_and_grad(state["X"], state["nact"], state["T"])
        net.adam_step()
        return {"loss": loss, "gW": net.gW, "gb": net.gb, "W": net.W, "b": net.b}
    return net.predict(state["X"], state["nact"])


# ---------------------------------------------------------------------- work
def _solve_work(g, precision, iters):
    """Per iteration: every terminal's value read; every other node's two
    reach lanes and its value written and read, and its place in the tree
    read; every slot's regret and average read and written in 64 bits and its
    strategy read and written."""
    T = precision // 8
    term = int((g.kind == gg.TERMINAL).sum())
    inner = g.n_nodes - term
    b = T * term + (6 * T + 4) * inner + (32 + 2 * T) * g.n_slots
    return {"bytes": float(iters * b), "flops": float(iters * 8 * g.n_edges)}


def _evaluate_work(g):
    """Terminal payoffs read; every other node's two reach lanes and three
    values (both best responses and the average) written and read, and its
    place in the tree read; the strategy read."""
    term = int((g.kind == gg.TERMINAL).sum())
    inner = g.n_nodes - term
    return {"bytes": float(8 * term + (80 + 4) * inner + 8 * g.n_slots), "flops": float(10 * g.n_edges)}


def work(case):
    kind = case["kind"]
    if kind == "solve":
        return _solve_work(_structure(case), case["precision"], case["iters"])
    if kind == "evaluate":
        return _evaluate_work(_structure(case))
    if kind in ("round", "serve"):
        total = {"bytes": 0.0, "flops": 0.0}
        rounds = 1 if kind == "round" else -(-case["iters"] // 25)
        for g in _batch_structures(case["n"], case["lo"], case["hi"], case["a"]):
            w, e = _solve_work(g, case.get("precision", 32), case["iters"]), _evaluate_work(g)
            for k in total:
                total[k] += w[k] + rounds * e[k]
        return total
    dims = [warmstart.F_IN, 256, 256, 256, mlp.N_OUT]
    weights = sum(i * o for i, o in zip(dims, dims[1:]))
    rows = case["rows"]
    if kind == "train":
        # rows and targets read; weights and both moments read and written,
        # gradients written
        return {"bytes": float(rows * 4 * (dims[0] + mlp.N_OUT + 1) + 28 * weights),
                "flops": float(2 * rows * (3 * weights - dims[0] * dims[1]))}
    return {"bytes": float(rows * 4 * (dims[0] + mlp.N_OUT + 1) + 2 * weights), "flops": float(2 * rows * weights)}


# ----------------------------------------------------------------- tolerance
# About four times what the path showed against `exact`, or (the network)
# against the same products of BF16 operands summed by torch. Regret matching
# turns a rounding difference in a near-zero regret into another strategy at
# that set, so the differences of 32-bit solves grow with the iterations:
# 5e-7 after 5 iterations of the random tree, 3e-6 after 50 of an endgame
# batch, 4e-5 after 100. In the network a last-bit difference flips BF16
# roundings and ReLU signs of later layers, more so with fewer rows.


def tolerance(case):
    kind = case["kind"]
    if kind == "solve":
        return {"rel": 1e-10} if case["precision"] == 64 else {"rel": 1e-5, "max": 2e-3}
    if kind == "evaluate":
        return {"rel": 1e-11}
    if kind in ("round", "serve"):
        return {"rel": 1e-10} if case.get("precision", 32) == 64 else {"rel": 1.6e-4, "max": 2e-2}
    if kind == "train":
        return {"rel": 3e-3, "max": 4e-2} if case["rows"] >= 2048 else {"rel": 2.5e-2, "max": 0.35}
    return {"rel": 1e-4, "max": 7e-3}


# --------------------------------------------------------- results in 64 bits
class _Levels:
    """A tabular game as one list of edges for each depth (torch, 64 bits)."""

    def __init__(self, g):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda x, d: torch.as_tensor(np.ascontiguousarray(x), device=dev).to(d)  # noqa: E731
        self.dev, self.n, self.pot = dev, g.n_nodes, g.pot
        kind = t(g.kind, torch.int64)
        begin, child = t(g.child_begin, torch.int64), t(g.child, torch.int64)
        iset = t(g.infoset, torch.int64)
        nact = t(g.iset_nact, torch.int64)
        first = torch.cumsum(nact, 0) - nact
        self.A, self.I = int(nact.sum()), len(nact)
        self.iset_of_slot = torch.repeat_interleave(torch.arange(self.I, device=dev), nact)
        self.player_of_slot = t(g.iset_player, torch.int64)[self.iset_of_slot]
        self.nact_of_slot = nact[self.iset_of_slot].double()
        self.first, self.nact = first, nact
        prob = t(g.chance_prob, torch.float64)
        self.payoff = torch.where(kind == 0, t(g.payoff, torch.float64), torch.zeros((), dtype=torch.float64, device=dev))
        self.levels = []
        front = torch.zeros(1, dtype=torch.int64, device=dev)
        while len(front):
            cnt = begin[front + 1] - begin[front]
            parent = torch.repeat_interleave(front, cnt)
            if not len(parent):
                break
            act = torch.arange(len(parent), device=dev) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            e = begin[parent] + act
            k = kind[parent]
            slot = torch.where(k >= 2, first[iset[parent].clamp(min=0)] + act, torch.full_like(act, -1))
            self.levels.append((parent, child[e], k, slot, prob[e]))
            front = child[e]

    def matched(self, x):
        """Regret matching of x per set, uniform where nothing is positive."""
        x = x.clamp(min=0.0)
        tot = torch.zeros(self.I, dtype=torch.float64, device=self.dev).index_add_(0, self.iset_of_slot, x)
        tot = tot[self.iset_of_slot]
        return torch.where(tot > 0, x / tot, 1.0 / self.nact_of_slot)

    def weight(self, lev, sigma):
        _, _, k, slot, p = lev
        return torch.where(k == 1, p, sigma[slot.clamp(min=0)])

    def reach(self, sigma):
        """Chance's, player 1's and player 2's reach of every node."""
        r = torch.ones(3, self.n, dtype=torch.float64, device=self.dev)
        for lev in self.levels:
            parent, c, k, _, _ = lev
            w = self.weight(lev, sigma)
            for q in range(3):
                r[q, c] = r[q, parent] * torch.where(k == q + 1, w, 1.0)
        return r

    def value(self, sigma):
        v = self.payoff.clone()
        for lev in reversed(self.levels):
            v.index_add_(0, lev[0], self.weight(lev, sigma) * v[lev[1]])
        return v

    def solve(self, iters, rule, order):
        """(average strategy, current strategy) after iters iterations."""
        z = lambda: torch.zeros(self.A, dtype=torch.float64, device=self.dev)  # noqa: E731
        R, S = z(), z()
        sigma = self.matched(R)
        for t in range(1, iters + 1):
            for upd in ([(0, 1)] if not order else [(0,), (1,)]):
                r, v = self.reach(sigma), self.value(sigma)
                inst, own = z(), z()
                for parent, c, k, slot, _ in self.levels:
                    for q in upd:
                        m = k == q + 2
                        h, s = parent[m], slot[m]
                        cf = r[0, h] * r[2 - q, h]
                        inst.index_add_(0, s, (1.0 if q == 0 else -1.0) * cf * (v[c[m]] - v[h]))
                        own.index_add_(0, s, r[1 + q, h] * sigma[s])
                mine = torch.zeros(self.A, dtype=torch.bool, device=self.dev)
                for q in upd:
                    mine |= self.player_of_slot == q
                new = R + inst
                if rule != 1:
                    new = new.clamp(min=0.0)
                R = torch.where(mine, new, R)
                S = S + own * float(t * t if rule == 2 else t)
                sigma = torch.where(mine, self.matched(R + inst if rule == 2 else R), sigma)
        return self.normalised(S), sigma

    def normalised(self, S):
        tot = torch.zeros(self.I, dtype=torch.float64, device=self.dev).index_add_(0, self.iset_of_slot, S)
        tot = tot[self.iset_of_slot]
        return torch.where(tot > 0, S / tot, 1.0 / self.nact_of_slot)

    def best_response(self, sigma):
        """(exploitability, player 1's best response value, player 2's, the
        value of sigma), all as payoffs to player 1."""
        r = self.reach(sigma)
        best = []
        for q in (0, 1):
            v = self.payoff.clone()
            for lev in reversed(self.levels):
                parent, c, k, slot, _ = lev
                m = k == q + 2
                w = self.weight(lev, sigma)
                if bool(m.any()):
                    Q = torch.zeros(self.A, dtype=torch.float64, device=self.dev)
                    Q.index_add_(0, slot[m], r[0, parent[m]] * r[2 - q, parent[m]] * v[c[m]])
                    Q = Q if q == 0 else -Q
                    top = torch.full((self.I,), -torch.inf, dtype=torch.float64, device=self.dev)
                    top.scatter_reduce_(0, self.iset_of_slot, Q, "amax")
                    at = torch.where(Q >= top[self.iset_of_slot], torch.arange(self.A, device=self.dev), self.A)
                    arg = torch.full((self.I,), self.A, dtype=torch.int64, device=self.dev)
                    arg.scatter_reduce_(0, self.iset_of_slot, at, "amin")
                    chosen = torch.zeros(self.A, dtype=torch.float64, device=self.dev)
                    chosen[arg] = 1.0
                    w = torch.where(m, chosen[slot.clamp(min=0)], w)
                v.index_add_(0, parent, w * v[c])
            best.append(float(v[0]))
        return 0.5 * (best[0] - best[1]), best[0], best[1], float(self.value(sigma)[0])


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        avg, cur = _Levels(_game(case, seed)).solve(case["iters"], case["rule"], case["order"])
        return {"average": avg, "current": cur}
    if kind == "evaluate":
        g = _game(case, seed)
        lv = _Levels(g)
        avg = torch.as_tensor(_some_average(g, seed), device=lv.dev)
        return list(lv.best_response(lv.normalised(avg))[1:])
    if kind in ("round", "serve"):
        if case["n"] * case["iters"] * (case["hi"] - case["lo"]) > 2.5e9:
            return None
        ex, avg = [], []
        for g in _batch(case, seed):
            lv = _Levels(g)
            a, _ = lv.solve(case["iters"], 0, 0)
            e = lv.best_response(a)
            ex.append(e if kind == "round" else e[0])
            avg.append(a)
        out = {"exploitability": np.array(ex), "average": torch.cat(avg)}
        if kind == "serve":
            out["iterations"] = None
        return out
    X, nact, T = _rows(case, seed)
    net = _network(seed)
    W, b = [w.double() for w in net.W], [x.double() for x in net.b]
    hs = [X.double()]
    for l in range(len(W)):
        z = hs[-1] @ W[l] + b[l]
        hs.append(z.clamp(min=0.0) if l < len(W) - 1 else z)
    mask = torch.arange(mlp.N_OUT, device=X.device) < nact[:, None]
    lp = torch.log_softmax(hs[-1].masked_fill(~mask, -torch.inf), 1)
    p = lp.exp()
    if kind == "predict":
        return p
    T = T.double()
    loss = float(-(T * lp.masked_fill(~mask, 0.0)).sum() / len(X))
    d = (p * T.sum(1, keepdim=True) - T) / len(X)
    gW, gb = [None] * len(W), [None] * len(W)
    for l in range(len(W) - 1, -1, -1):
        gW[l], gb[l] = hs[l].T @ d, d.sum(0)
        if l:
            d = (d @ W[l].T) * (hs[l] > 0)
    def stepped(x, g, m, v):
        m, v = 0.9 * m.double() + 0.1 * g, 0.999 * v.double() + 0.001 * g * g
        m, v = m / (1.0 - 0.9 ** (STEPS + 1)), v / (1.0 - 0.999 ** (STEPS + 1))
        return x - 1e-3 * m / (v.sqrt() + 1e-8)

    return {"loss": loss, "gW": gW, "gb": gb, "W": [stepped(*t) for t in zip(W, gW, net.mW, net.vW)],
            "b": [stepped(*t) for t in zip(b, gb, net.mb, net.vb)]}
