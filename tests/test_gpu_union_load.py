"""Batches loaded as one union: games of every small size next to each other,
games without and with dummies, sparse priorities (the general path), both
offset widths, and a batch of two chunks, each game against the oracle or its
own pg_solve."""
import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300 import gen
from paper_1705_02313_gb300.gen import Game

pytestmark = pytest.mark.gpu

KEYS = ["win", "sigma", "tau", "val_class", "val_depth", "val_rank"]


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import pg
    return pg


@pytest.fixture(scope="module")
def ctx(pg):
    c = pg.pg_ctx_create(0)
    yield c
    pg.pg_ctx_destroy(c)


def buffers(n):
    return dict(win=np.empty(n, np.uint8), val_class=np.empty(n, np.int8), dummy_sigma=np.empty(n, np.int8),
                **{k: np.empty(n, np.int32) for k in ("sigma", "tau", "val_depth", "val_rank")})


def check(pg, ctx, games):
    vb, eb, *arrays = pg.pack_games(games)
    out = buffers(int(vb[-1]))
    r = pg.pg_solve_batch(ctx, len(games), vb, eb, *arrays, **out)
    for i, g in enumerate(games):
        gp, res, want = o2.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)
        assert (r["major"][i], r["inner"][i]) == (want["major"], want["inner"]), i
        for k in KEYS:
            assert np.array_equal(out[k][vb[i] : vb[i + 1]], np.asarray(want[k])), (i, k)
        d0, d1 = r["dummy_base"][i], r["dummy_base"][i + 1]
        assert np.array_equal(out["dummy_sigma"][d0:d1], res["strat"][g.n :] != gp["n"]), i


def one_owner(n, odd, seed):
    g = gen.random_game(n, 1, 3, seed=seed)
    g.owner[:] = odd
    return g


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("spread", [1, 1000, 40_000_000])  # the last: too sparse for the union's bitmaps
def test_small_games(pg, ctx, wide, spread):
    games = [gen.random_game(n, 1, 4, seed=n) for n in [1, 1, 2, 3, 31, 32, 33, 255, 257, 1000, 5]]
    games += [one_owner(40, 0, 1), one_owner(40, 1, 2), one_owner(1, 1, 3), gen.ladder_game(2, 4)]
    for g in games:
        g.pri[:] = np.minimum(g.pri.astype(np.int64) * spread, 2**31 - 4000) - (g.pri.size - 1 - g.pri)
        assert np.unique(g.pri).size == g.n
        g.pri -= min(0, g.pri.min())
    pg.pg_set_wide_offsets(ctx, wide)
    try:
        check(pg, ctx, games)
    finally:
        pg.pg_set_wide_offsets(ctx, False)


def test_two_chunks(pg, ctx):
    games = [gen.native_random_game(34_000_000, 4, 4, seed=s) for s in (1, 2)]
    vb, eb, *arrays = pg.pack_games(games)
    out = buffers(int(vb[-1]))
    r = pg.pg_solve_batch(ctx, 2, vb, eb, *arrays, **out)
    for i, g in enumerate(games):
        want = pg.solve_arrays(ctx, g.n, *g.arrays())
        assert (r["major"][i], r["inner"][i]) == (want["major"], want["inner"])
        for k in KEYS:
            assert np.array_equal(out[k][vb[i] : vb[i + 1]], want[k]), k
        assert np.array_equal(out["dummy_sigma"][r["dummy_base"][i] : r["dummy_base"][i + 1]], want["dummy_sigma"])
