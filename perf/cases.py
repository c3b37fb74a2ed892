"""The work that users of this library have it do, as measurable cases.

Each case goes through the public entry points of ``paper_1705_02313_gb300.pg``
with inputs made from a seed: whole solves (load, Algorithm 1, results) of
random, ladder and few-priority games from the smallest call to the largest
workload, best responses and valuations of a loaded game, the allocation-free
valuation, a batch, and a burst of requests to a server.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` makes what a program holds before the call, ``run(state)``
is one call, ``work(case)`` the bytes that it cannot do without, and
``exact(case, seed)`` the outputs as plain numpy gives them, where it can.
"""
import math

import numpy as np
import torch

from paper_1705_02313_gb300 import gen, pg

DEVICE = "cuda"


def listed():
    return [
        # the smallest call: one small game from host arrays to host results, load and solve; launches and
        # waits are all of it
        dict(name="random-1k-host", kind="solve", shape="random", n=1_000, dmin=1, dmax=4, p_odd=0.5, host=True,
             reset=False),
        # a small verification-sized game, device arrays, an odd size
        dict(name="random-30k", kind="solve", shape="random", n=30_011, dmin=2, dmax=6, p_odd=0.5, host=False,
             reset=False),
        # the 1M-vertex random workload: every array of the loop fits the L2 cache
        dict(name="random-1m", kind="solve", shape="random", n=1_000_000, dmin=2, dmax=8, p_odd=0.5, host=False,
             reset=False),
        # the headline workload: the 10M-vertex random game, loaded and solved on the device
        dict(name="random-10m", kind="solve", shape="random", n=10_000_000, dmin=2, dmax=5, p_odd=0.5, host=False,
             reset=False),
        # the 10M-vertex ladder: long successor chains, the most valuations of the named workloads
        dict(name="ladder-10m", kind="solve", shape="ladder", n=10_000_000, dmin=2, dmax=2, p_odd=0.5, host=False,
             reset=False),
        # verification games have two to four priorities: count-vector mode, with the counts among the results
        dict(name="levels-3m-4pri", kind="solve", shape="levels", n=3_000_017, dmin=2, dmax=5, p_odd=0.5, host=False,
             reset=False),
        # Odd's best response to a good Even strategy from a cold start, on a loaded game
        dict(name="response-1m", kind="response", n=1_000_003, dmin=2, dmax=5, p_odd=0.5),
        # the valuation of a profile under study, with the dominant priorities of its cycles
        dict(name="valuate-4m", kind="valuate", shape="random", n=4_000_037, dmin=2, dmax=5, p_odd=0.5),
        # the valuation of one long play through all vertices: no parallelism along the play itself
        dict(name="chain-10m", kind="valuate", shape="chain", n=10_000_000, dmin=1, dmax=1, p_odd=0.0),
        # the allocation-free valuation inside a latency-bound loop
        dict(name="static-100k", kind="static", n=100_003, p_sink=0.3),
        # many games of mixed sizes solved together
        dict(name="batch-256", kind="batch", count=256, lo=1_000, hi=100_000, dmin=2, dmax=6, p_odd=0.5),
        # a burst of requests to a server from host arrays, polled and fetched
        dict(name="serve-8", kind="serve", count=8, lo=10_000, hi=1_000_000, dmin=2, dmax=6, p_odd=0.5),
    ]


def _between(rng, lo, hi):
    """An integer log-uniform in [lo, hi]."""
    return max(lo, min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    degrees = [(1, 4), (2, 5), (2, 6), (2, 8)]
    kind = rng.choice(["solve", "solve", "solve", "solve", "response", "valuate", "static", "batch", "serve"])
    dmin, dmax = rng.choice(degrees)
    p_odd = rng.choice([0.4, 0.5, 0.5, 0.6])
    if kind == "solve":
        shape = rng.choice(["random", "random", "ladder", "levels"])
        n = _between(rng, 500, {"random": 5_000_000, "ladder": 5_000_000, "levels": 2_000_000}[shape])
        # SI-Reset restarts Odd after every Even switch and takes about twice as many valuations
        reset = n <= 1_000_000 and rng.random() < 0.15
        return dict(kind=kind, shape=shape, n=n, dmin=2 if shape == "ladder" else dmin,
                    dmax=2 if shape == "ladder" else dmax, p_odd=p_odd, host=rng.random() < 0.3, reset=reset)
    if kind == "response":
        return dict(kind=kind, n=_between(rng, 1_000, 4_000_000), dmin=dmin, dmax=dmax, p_odd=p_odd)
    if kind == "valuate":
        if rng.random() < 0.4:
            return dict(kind=kind, shape="chain", n=_between(rng, 1_000, 8_000_000), dmin=1, dmax=1, p_odd=0.0)
        return dict(kind=kind, shape="random", n=_between(rng, 1_000, 6_000_000), dmin=dmin, dmax=dmax, p_odd=p_odd)
    if kind == "static":
        return dict(kind=kind, n=_between(rng, 64, 1 << 18), p_sink=rng.choice([0.05, 0.3, 0.6]))
    if kind == "batch":
        lo = _between(rng, 200, 5_000)
        return dict(kind=kind, count=rng.randint(8, 200), lo=lo, hi=min(100_000, lo * rng.randint(2, 40)), dmin=dmin, dmax=dmax,
                    p_odd=p_odd)
    lo = _between(rng, 1_000, 50_000)
    return dict(kind=kind, count=rng.randint(2, 8), lo=lo, hi=lo * rng.randint(2, 20), dmin=dmin, dmax=dmax,
                p_odd=p_odd)


# ---------------------------------------------------------------------------
# inputs

def _up(x):
    return torch.from_numpy(x).to(DEVICE)


def _random(case, seed, levels=0):
    return gen.native_random_game(case["n"], case["dmin"], case["dmax"], seed=seed, p_odd=case["p_odd"],
                                  levels=levels).arrays()


def _games(case, seed):
    """The games of a batch or a burst; their sizes belong to the case."""
    sizes = gen.log_uniform_sizes(case["count"], case["lo"], case["hi"])
    return [gen.native_random_game(int(n), case["dmin"], case["dmax"], seed=gen.batch_seed(seed * 4096 + i),
                                   p_odd=case["p_odd"]) for i, n in enumerate(sizes)]


def _ladder(case, seed):
    """Vertex i has one back edge to j < i and the edge to i + 1 (the first and
    the last vertex only one of the two); owners and priorities are random."""
    n = case["n"]
    r = torch.Generator(device=DEVICE)
    r.manual_seed(seed)
    i = torch.arange(n, device=DEVICE, dtype=torch.int64)
    off = torch.empty(n + 1, device=DEVICE, dtype=torch.int32)
    off[0] = 0
    off[1:n] = (2 * i[: n - 1] + 1).int()
    off[n] = 2 * n - 2
    back = (torch.rand(n, device=DEVICE, dtype=torch.float64, generator=r) * i.double()).long().clamp_(min=0)
    both = torch.stack([torch.minimum(back, (i - 1).clamp_(min=0)), i + 1], 1).reshape(-1)
    tgt = both[1 : 2 * n - 1].int().contiguous()
    own = (torch.rand(n, device=DEVICE, generator=r) < case["p_odd"]).to(torch.uint8)
    pri = torch.randperm(n, device=DEVICE, generator=r).int()
    return off, tgt, own, pri


def _arrays(case, seed):
    """The game's four arrays: device tensors, or host arrays for a host case."""
    if case["shape"] == "ladder":
        a = _ladder(case, seed)
        return tuple(x.cpu().numpy() for x in a) if case.get("host") else a
    a = _random(case, seed, levels=4 if case["shape"] == "levels" else 0)
    return a if case.get("host") else tuple(_up(x) for x in a)


def _chain(case, seed):
    """An all-Even game whose profile is one play through every vertex in a
    random order: (offsets, targets, owner, priorities, sigma) on the host."""
    n = case["n"]
    r = np.random.default_rng(seed)
    order = r.permutation(n).astype(np.int32)
    sigma = np.full(n, -1, np.int32)
    sigma[order[:-1]] = order[1:]
    tgt = np.where(sigma < 0, np.arange(n, dtype=np.int32), sigma).astype(np.int32)
    return (np.arange(n + 1, dtype=np.int32), tgt, np.zeros(n, np.uint8), r.permutation(n).astype(np.int32), sigma)


def _successors(case, seed):
    """A successor function over priority ranks (n names the sink) and the
    priorities' parities, on the host."""
    n = case["n"]
    r = np.random.default_rng(seed)
    succ = np.where(r.random(n) < case["p_sink"], n, r.integers(0, n, n)).astype(np.int32)
    return succ, (r.random(n) < 0.5).astype(np.uint8)


class _Owned:
    """A context, and the game or server that lives in it, freed with it."""

    def __init__(self, server=None):
        self.server = server
        self.game = None
        self.ctx = None
        if server is None:
            self.ctx = pg.pg_ctx_create(0)
            pg.pg_set_stream(self.ctx, torch.cuda.current_stream())

    def __del__(self):
        if self.server is not None:
            pg.pg_server_destroy(self.server)
        if self.game is not None:
            pg.pg_game_free(self.game)
        if self.ctx is not None:
            pg.pg_ctx_destroy(self.ctx)


def _values(n, device=DEVICE):
    return dict(val_class=torch.zeros(n, dtype=torch.int8, device=device),
                val_depth=torch.zeros(n, dtype=torch.int32, device=device),
                val_rank=torch.zeros(n, dtype=torch.int32, device=device))


def _results(n, dummies, device=DEVICE):
    return dict(win=torch.zeros(n, dtype=torch.uint8, device=device),
                sigma=torch.zeros(n, dtype=torch.int32, device=device),
                tau=torch.zeros(n, dtype=torch.int32, device=device), **_values(n, device),
                dummy_sigma=torch.zeros(dummies, dtype=torch.int8, device=device))


def _load(s, arrays):
    return pg.pg_load_csr(s["own"].ctx, s["case"]["n"], arrays[1].shape[0], *arrays)


def _random_edges(off, tgt, seed):
    """One edge of every vertex, at random."""
    r = torch.Generator(device=DEVICE)
    r.manual_seed(seed)
    deg = off[1:] - off[:-1]
    pick = (torch.rand(deg.shape[0], device=DEVICE, generator=r) * deg).int()
    return tgt[(off[:-1] + torch.minimum(pick, deg - 1)).long()].contiguous(), r


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        games = _games(case, seed)
        room = 2 * sum(g.n for g in games) + 1024  # every vertex of a game may have a dummy; one sink a game
        server = pg.pg_server_create(0, max_vertices=room, max_edges=room + sum(g.m for g in games))
        return dict(case=case, own=_Owned(server), games=games, dummies=[np.zeros(g.n, np.int8) for g in games])
    s = dict(case=case, own=_Owned())
    if kind == "batch":
        vb, eb, off, tgt, own, pri = pg.pack_games(_games(case, seed))
        s.update(vb=vb, eb=eb, arrays=tuple(_up(x) for x in (off, tgt, own, pri)),
                 out=_results(int(vb[-1]), int(vb[-1])))
        return s
    n = case["n"]
    if kind == "static":
        succ, odd = _successors(case, seed)
        s.update(succ=_up(succ), odd=_up(odd), out=_values(n))
        return s
    if kind == "solve":
        s.update(arrays=_arrays(case, seed))
        if case["host"]:
            s.update(out={k: v.numpy() for k, v in _results(n, n, "cpu").items()})
            if case["shape"] == "levels":
                s.update(counts=np.zeros(5 * n, np.int32))
        else:
            s.update(out=_results(n, n))
            if case["shape"] == "levels":
                s.update(counts=torch.zeros(5 * n, dtype=torch.int32, device=DEVICE))
        return s
    if kind == "response":
        off, tgt, own, pri = (_up(x) for x in _random(case, seed))
        s["own"].game = game = _load(s, (off, tgt, own, pri))
        k = pg.pg_game_info(game)[2]
        good = _results(n, max(k, 1))
        pg.pg_solve(s["own"].ctx, game, **good)
        s.update(sigma=good["sigma"], dummies=good["dummy_sigma"], cold=tgt[off[:-1].long()].contiguous(),
                 tau=torch.zeros(n, dtype=torch.int32, device=DEVICE), out=_values(n))
        return s
    if case["shape"] == "chain":
        off, tgt, own, pri, sigma = (_up(x) for x in _chain(case, seed))
        tau = torch.full_like(sigma, -1)
    else:
        off, tgt, own, pri = (_up(x) for x in _random(case, seed))
        tau, r = _random_edges(off, tgt, seed)
        sink = torch.rand(n, device=DEVICE, generator=r) < 0.3
        sigma = torch.where(sink, torch.full_like(tau, -1), tau)
    s["own"].game = _load(s, (off, tgt, own, pri))
    s.update(sigma=sigma, tau=tau, out=dict(_values(n), dom=torch.zeros(n, dtype=torch.int32, device=DEVICE)))
    return s


def _solve(s):
    case, ctx = s["case"], s["own"].ctx
    game = _load(s, s["arrays"])
    try:
        out = dict(s["out"])
        if case["shape"] == "levels":
            d = len(pg.pg_game_levels(game))
            out["val_counts"] = s["counts"][: case["n"] * d]
        major, inner = pg.pg_solve(ctx, game, reset_tau=case["reset"], **out)
    finally:
        pg.pg_game_free(game)
    # the buffers are sized for any game of this many vertices: entries beyond its dummies and levels stay zero
    return dict(s["out"], counts=s.get("counts"), major=major, inner=inner)


def _serve(s):
    server, games = s["own"].server, s["games"]
    for tag, g in enumerate(games):
        pg.pg_server_submit(server, g.n, g.m, *g.arrays(), tag)
    got = [None] * len(games)
    left = len(games)
    while left:
        for d in pg.pg_server_poll(server, timeout_ms=1000):
            tag = d["tag"]
            got[tag] = pg.pg_server_fetch(server, tag, d["n"], d["k"])
            s["dummies"][tag][: d["k"]] = got[tag]["dummy_sigma"]
            got[tag]["dummy_sigma"] = s["dummies"][tag]
            left -= 1
    return got


def run(s):
    case = s["case"]
    kind, ctx, game = case["kind"], s["own"].ctx, s["own"].game
    if kind == "solve":
        return _solve(s)
    if kind == "serve":
        return _serve(s)
    if kind == "batch":
        r = pg.pg_solve_batch(ctx, case["count"], s["vb"], s["eb"], *s["arrays"], **s["out"])
        return dict(s["out"], major=r["major"], inner=r["inner"], status=r["status"], dummy_base=r["dummy_base"])
    if kind == "static":
        rc = pg.pg_valuate_static(case["n"], s["succ"], s["odd"], stream=torch.cuda.current_stream(), **s["out"])
        return dict(s["out"], rc=rc)
    if kind == "response":
        s["tau"].copy_(s["cold"])
        iters = pg.pg_best_response(ctx, game, s["sigma"], s["tau"], s["dummies"], **s["out"])
        return dict(s["out"], tau=s["tau"], iters=iters)
    rc = pg.pg_valuate(ctx, game, s["sigma"], s["tau"], **s["out"])
    return dict(s["out"], rc=rc)


# ---------------------------------------------------------------------------
# what a pass cannot do without, and its outputs from plain numpy

def work(case):
    """The call's arrays read once and its results written once. The passes of
    the iterations between them depend on the game and are not counted."""
    kind = case["kind"]
    results = 18  # winner, two strategies, class, depth and rank of a vertex
    if kind in ("batch", "serve"):
        lo, hi = case["lo"], case["hi"]
        n = case["count"] * ((hi - lo) / math.log(hi / lo) if hi > lo else lo)
    else:
        n = case["n"]
    m = n * (case["dmin"] + case["dmax"]) / 2 if "dmin" in case else 0
    if kind == "static":
        return dict(bytes=5 * n + 9 * n, flops=0)
    if kind == "valuate":
        return dict(bytes=8 * n + 13 * n, flops=0)
    if kind == "response":
        # both strategies in, Odd's edges once, its strategy and the valuation out
        return dict(bytes=8 * n + 4 * m * case["p_odd"] + 4 * n + 9 * n, flops=0)
    counts = 20 if case.get("shape") == "levels" else 0
    return dict(bytes=9 * n + 4 * m + (results + counts) * n, flops=0)


def _plays(succ):
    """(infinite, vertices before the sink or -1) of every vertex under succ,
    whose sink is len(succ), by pointer doubling."""
    n = succ.shape[0]
    at = np.append(succ.astype(np.int64), n)
    steps = np.append(np.ones(n, np.int64), 0)
    for _ in range(n.bit_length()):
        steps = steps + steps[at]
        at = at[at]
    top = at[:n] != n
    return top, np.where(top, -1, steps[:n])


def exact(case, seed):
    """Class and depth of every vertex where the play is given; ranks and whole
    solves have no short form in plain numpy."""
    if case["kind"] == "static":
        top, depth = _plays(_successors(case, seed)[0])
        return dict(val_class=top.astype(np.int8), val_depth=depth.astype(np.int32), val_rank=None, rc=None)
    if case["kind"] == "valuate" and case["shape"] == "chain":
        n = case["n"]
        sigma = _chain(case, seed)[4]
        top, depth = _plays(np.where(sigma < 0, n, sigma))
        return dict(val_class=top.astype(np.int8), val_depth=depth.astype(np.int32), val_rank=None,
                    dom=np.full(n, -1, np.int32), rc=0)
    return None
