"""Valuations of small games in one cluster (csrc/pg_small.cu): pg_valuate and
pg_valuate_static around the sizes of a block and of the cluster, forests of
every fan-out class, long chains and cycles, against the oracle."""
import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300.gen import Game

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import pg
    return pg


def profile(n, shape, seed):
    """A successor function over ids 0..n-1 (n: the sink)."""
    r = np.random.default_rng(seed)
    if shape == "random":
        return np.where(r.random(n) < 0.2, n, r.integers(0, n, n)).astype(np.int32)
    if shape == "rising":  # each vertex to one of the next few: deep chains
        return np.minimum(np.arange(n) + r.integers(1, 4, n), n).astype(np.int32)
    if shape == "fans":  # parents with 3, 20, 300 and (from 6,000 vertices on) over 4,096 children
        s = np.full(n, n, np.int32)
        at = 0
        for k in [3, 20, 300, 5000] * 2:
            top = n - 1 - at
            if at + k + 1 < n // 2:
                s[at : at + k] = top
                at += k
        return s
    s = np.empty(n, np.int32)  # one play through all vertices, then a cycle
    order = r.permutation(n)
    s[order[:-1]] = order[1:]
    s[order[-1]] = order[n // 2]
    return s


def oracle(succ, odd):
    n = succ.size
    pri = 2 * np.arange(n, dtype=np.int32) + odd  # id = priority rank
    val = o2.valuate(dict(n=n, pri=pri), succ)
    top = val["cls"] != o2.FIN
    return top.astype(np.int8), np.where(top, -1, val["depth"]), np.where(top, o2.INT32_MAX, val["rank"]), pri, val


@pytest.mark.parametrize("n", [1, 2, 31, 1023, 1024, 1025, 8193, 20000, 65537, 262144])
@pytest.mark.parametrize("shape", ["random", "rising", "fans", "cycle"])
def test_valuations(pg, n, shape):
    import torch
    succ = profile(n, shape, n)
    odd = (np.random.default_rng(n + 1).random(n) < 0.5).astype(np.uint8)
    cls, depth, rank, pri, val = oracle(succ, odd)
    dev = [torch.from_numpy(x).cuda() for x in (succ, odd)]
    out = [torch.zeros(n, dtype=t, device="cuda") for t in (torch.int8, torch.int32, torch.int32)]
    for _ in range(2):
        pg.pg_valuate_static(n, *dev, *out)
        for got, want in zip(out, (cls, depth, rank)):
            assert np.array_equal(got.cpu().numpy(), want)
    if n >= 262144:
        return
    # the same profile as an all-Even game's strategy (a self-loop stands in for the sink's vertices)
    tgt = np.where(succ == n, np.arange(n), succ).astype(np.int32)
    g = Game(n, np.arange(n + 1, dtype=np.int32), tgt, np.zeros(n, np.uint8), pri)
    sigma = np.where(succ == n, -1, succ).astype(np.int32)
    ctx = pg.pg_ctx_create(0)
    game = pg.pg_load_csr(ctx, n, n, *g.arrays())
    try:
        o = dict(val_class=np.empty(n, np.int8), val_depth=np.empty(n, np.int32), val_rank=np.empty(n, np.int32),
                 dom=np.empty(n, np.int32))
        pg.pg_valuate(ctx, game, sigma, np.full(n, -1, np.int32), **o)
    finally:
        pg.pg_game_free(game)
        pg.pg_ctx_destroy(ctx)
    assert np.array_equal(o["val_class"], cls) and np.array_equal(o["val_depth"], depth)
    assert np.array_equal(o["val_rank"], rank)
    assert np.array_equal(o["dom"], np.where(cls == 1, val["dom"], -1))
