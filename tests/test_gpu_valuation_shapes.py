"""One-launch valuations (csrc/pg_small.cu) where their rules change: what the
cluster's threads and one block per SM hold at once, parents with as many
children as a warp orders, and long chains, which a second round of threads or
unequal lanes would double. Values against the oracle, times against the
separate kernels (which a context with timing enabled runs)."""
import time

import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300.gen import Game

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import build, pg as _pg
    build.build()
    return _pg


@pytest.fixture
def ctx(pg):
    c = pg.pg_ctx_create(0, tuning=False)
    yield c
    pg.pg_ctx_destroy(c)


def profile(n, shape, seed):
    """A successor function over ids 0..n-1 (n: the sink)."""
    r = np.random.default_rng(seed)
    v = np.arange(n)
    if shape == "play":  # one play through all vertices in a random order
        s = np.full(n, n, np.int64)
        order = r.permutation(n)
        s[order[:-1]] = order[1:]
    elif shape == "runs":  # runs of 50 rising vertices
        s = np.where(v % 50 == 49, n, v + 1)
    elif shape == "kids":  # parents at the top with 31 .. 130 children each, most of these below a child of theirs
        s = np.full(n, n, np.int64)
        at, top = 0, n - 1
        for k in [31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 130] * (n // 2000 + 1):
            if at + k >= top - 1:
                break
            s[at:at + k] = top
            if at:
                s[top] = r.integers(top + 1, n) if top + 1 < n and r.random() < 0.3 else n
            at, top = at + k, top - 1
    else:
        s = np.where(r.random(n) < 0.3, n, r.integers(0, n, n))
    return s.astype(np.int32)


def game_of(succ, odd):
    """The profile as an all-Even game's strategy (a self-loop stands in for the sink's vertices)."""
    n = succ.size
    pri = (2 * np.arange(n) + odd).astype(np.int32)  # id = priority rank
    tgt = np.where(succ == n, np.arange(n), succ).astype(np.int32)
    return Game(n, np.arange(n + 1, dtype=np.int32), tgt, np.zeros(n, np.uint8), pri), \
        np.where(succ == n, -1, succ).astype(np.int32)


@pytest.mark.parametrize("n", [16_383, 16_384, 155_647, 155_648, 200_003, 262_144])
@pytest.mark.parametrize("shape", ["play", "runs", "kids", "random"])
def test_values(pg, ctx, n, shape):
    import torch
    succ = profile(n, shape, n)
    odd = (np.random.default_rng(n + 1).random(n) < 0.5).astype(np.uint8)
    g, sigma = game_of(succ, odd)
    val = o2.valuate(dict(n=n, pri=g.pri), succ)
    top = val["cls"] != o2.FIN
    cls, depth = top.astype(np.int8), np.where(top, -1, val["depth"])
    rank = np.where(top, o2.INT32_MAX, val["rank"])
    dev = [torch.from_numpy(x).cuda() for x in (succ, odd)]
    out = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.int8, torch.int32, torch.int32)]
    pg.pg_valuate_static(n, *dev, *out)
    for got, want in zip(out, (cls, depth, rank)):
        assert np.array_equal(got.cpu().numpy(), want)
    game = pg.pg_load_csr(ctx, n, g.m, *g.arrays())
    try:
        o = dict(val_class=np.empty(n, np.int8), val_depth=np.empty(n, np.int32), val_rank=np.empty(n, np.int32))
        pg.pg_valuate(ctx, game, sigma, np.full(n, -1, np.int32), **o)
    finally:
        pg.pg_game_free(game)
    for k, want in (("val_class", cls), ("val_depth", depth), ("val_rank", rank)):
        assert np.array_equal(o[k], want), k


@pytest.mark.parametrize("shape", ["play", "runs"])
def test_long_chains_are_not_slower_than_by_the_separate_kernels(pg, ctx, shape):
    import torch
    n = 260_000
    succ = profile(n, shape, 3)
    g, sigma = game_of(succ, np.zeros(n, np.uint8))
    game = pg.pg_load_csr(ctx, n, g.m, *g.arrays())
    sig = torch.from_numpy(sigma).cuda()
    o = dict(val_class=torch.empty(n, dtype=torch.int8, device="cuda"),
             val_rank=torch.empty(n, dtype=torch.int32, device="cuda"))
    took = {}
    try:
        for timing in (0, 1):
            pg.pg_set_timing(ctx, timing)
            ts = []
            for _ in range(25):
                t = time.perf_counter()
                pg.pg_valuate(ctx, game, sig, None, None, **o)
                ts.append(time.perf_counter() - t)
            took[timing] = sorted(ts)[12]
    finally:
        pg.pg_game_free(game)
    assert took[0] <= 1.05 * took[1], took
