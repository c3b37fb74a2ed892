"""Batches whose games run their loops in a cluster each (csrc/pg_inc.cu): games
around the sizes of a block and of both block sizes, few and many games (every
cluster size), long ladders, iteration caps, and batches with a deep game that
the lockstep loop finishes, each game against the oracle."""
import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300 import gen

pytestmark = pytest.mark.gpu

KEYS = ["win", "sigma", "tau", "val_class", "val_depth", "val_rank"]


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import pg
    return pg


@pytest.fixture()
def ctx(pg):
    c = pg.pg_ctx_create(0)
    yield c
    pg.pg_ctx_destroy(c)


def solve(pg, ctx, games, max_inner=0):
    vb, eb, *arrays = pg.pack_games(games)
    n = int(vb[-1])
    out = dict(win=np.empty(n, np.uint8), val_class=np.empty(n, np.int8),
               **{k: np.empty(n, np.int32) for k in ("sigma", "tau", "val_depth", "val_rank")})
    r = pg.pg_solve_batch(ctx, len(games), vb, eb, *arrays, max_inner=max_inner, **out)
    return vb, r, out


def check(pg, ctx, games):
    vb, r, out = solve(pg, ctx, games)
    for i, g in enumerate(games):
        _, _, want = o2.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)
        assert (r["major"][i], r["inner"][i]) == (want["major"], want["inner"]), (i, g.n)
        for k in KEYS:
            assert np.array_equal(out[k][vb[i] : vb[i + 1]], np.asarray(want[k])), (i, g.n, k)
    assert r["iterations"] == r["inner"].max()


def some(sizes, seed):
    return [gen.random_game(n, 1 + i % 2, 2 + i % 4, seed=seed + i, p_odd=[0.5, 0.2, 0.8][i % 3])
            for i, n in enumerate(sizes)]


@pytest.mark.parametrize("sizes", [[1], [40_000], [12_000, 14_000, 16_383, 90_000], [100] * 600, [100] * 700,
                                   [255, 256, 1023, 1024, 1025, 2048] * 20, [17_000] * 20, [30_000] * 5 + [2] * 9,
                                   [9_000] * 100])
def test_random_games(pg, ctx, sizes):
    check(pg, ctx, some(sizes, len(sizes)))


def test_ladders(pg, ctx):
    check(pg, ctx, [gen.ladder_game(n, n) for n in (2, 3, 1000, 15_000, 33_000, 60_000)])


def test_with_a_deep_game(pg, ctx):
    from test_gpu_deep import climbing_game
    check(pg, ctx, some([5000, 300, 20_000], 3) + [climbing_game(3000, 1, 0.05)])


@pytest.mark.parametrize("cap", [1, 4])
def test_iteration_cap(pg, ctx, cap):
    games = some([3000, 20_000, 1, 150], 11)
    vb, eb, *arrays = pg.pack_games(games)
    ends = []
    for graphs in (True, False):  # clusters, and the lockstep loop
        pg.pg_set_graphs(ctx, graphs)
        n = int(vb[-1])
        out = {k: np.full(n, -7, np.int32) for k in ("sigma", "tau", "val_depth", "val_rank")}
        try:
            r = pg.pg_solve_batch(ctx, len(games), vb, eb, *arrays, max_inner=cap, **out)
            ends.append((list(r["inner"]), list(r["major"]), list(r["status"]), out))
        except pg.PgError as e:
            ends.append((e.args, out))
    assert ends[0][:-1] == ends[1][:-1]
    assert all(np.array_equal(ends[0][-1][k], ends[1][-1][k]) for k in ends[0][-1])
