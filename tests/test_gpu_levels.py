"""Forests with few roots (csrc/pg_level.cuh): valuations of games past the small
games' path whose forests have few roots, below and above the cutover depth,
with cycles and with parents of every fan-out class, against the oracle."""
import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300.gen import Game

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import pg
    return pg


def profile(n, shape, r):
    """A successor function over ids 0..n-1 (n: the sink)."""
    ids = np.arange(n)
    order = r.permutation(n)
    s = np.empty(n, np.int64)
    if shape in ("play", "cycle"):  # through all vertices in random order, then to the sink or back into the play
        s[order[:-1]] = order[1:]
        s[order[-1]] = n if shape == "play" else order[n // 2]
    elif shape == "both":  # a play and a cycle
        s[order[:-1]] = order[1:]
        s[order[n // 3]] = n
        s[order[-1]] = order[n // 2]
    elif shape == "hub":  # nearly every vertex a child of one, the rest in chains of 100 above it
        s[:] = n - 101
        s[n - 101 :] = np.arange(n - 100, n + 1)
    elif shape == "fans":  # 40 levels of parents with 2 to 9,000 children each
        s = np.minimum(ids + 1 + r.integers(0, 9000, n) ** 2 // 9000, n)
        s[ids >= n - 40 * 4000] = np.minimum(((ids[ids >= n - 40 * 4000] // 4000) + 1) * 4000, n)
        s[: n - 40 * 4000] = n - 40 * 4000 + r.integers(0, 4000, n - 40 * 4000)
    elif shape == "ladder":  # two chains of 50 levels over 2^18 leaves
        s[:] = n - 100 + r.integers(0, 2, n)
        top = ids >= n - 100
        s[top] = np.minimum(ids[top] + 2, n)
    return s.astype(np.int32)


@pytest.mark.parametrize("n", [262145, 262144 + 4 * 155648 + 33])
@pytest.mark.parametrize("shape", ["play", "cycle", "both", "hub", "fans", "ladder"])
@pytest.mark.parametrize("deep_cut", [0, 1, 127, 128])
def test_deep_forests(pg, n, shape, deep_cut):
    r = np.random.default_rng(n)
    succ = profile(n, shape, r)
    pri = (2 * np.arange(n) + (r.random(n) < 0.5)).astype(np.int32)  # id = priority rank
    val = o2.valuate(dict(n=n, pri=pri), succ)
    top = val["cls"] != o2.FIN
    tgt = np.where(succ == n, np.arange(n), succ).astype(np.int32)  # (a self-loop stands in for the sink's vertices)
    g = Game(n, np.arange(n + 1, dtype=np.int32), tgt, np.zeros(n, np.uint8), pri)
    sigma = np.where(succ == n, -1, succ).astype(np.int32)
    ctx = pg.pg_ctx_create(0)
    if deep_cut:
        pg.pg_set_tuning(ctx, deep_cut=deep_cut, ruler_bits=0)
    game = pg.pg_load_csr(ctx, n, n, *g.arrays())
    try:
        for _ in range(2):
            o = dict(val_class=np.empty(n, np.int8), val_depth=np.empty(n, np.int32), val_rank=np.empty(n, np.int32),
                     dom=np.empty(n, np.int32))
            pg.pg_valuate(ctx, game, sigma, np.full(n, -1, np.int32), **o)
            assert np.array_equal(o["val_class"], top.astype(np.int8))
            assert np.array_equal(o["val_depth"], np.where(top, -1, val["depth"]))
            assert np.array_equal(o["val_rank"], np.where(top, o2.INT32_MAX, val["rank"]))
            assert np.array_equal(o["dom"], np.where(top, val["dom"], -1))
    finally:
        pg.pg_game_free(game)
        pg.pg_ctx_destroy(ctx)
