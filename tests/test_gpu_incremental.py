"""Incremental iterations (csrc/pg_inc.cu) against the oracle: games below and
above the size that one launch solves whole, around the thread counts of its
cluster, with many predecessors on a few vertices (closures that give up),
repeated edges and self-loops."""
import numpy as np
import pytest

from oracle import o2, o3
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


def hub_game(n, hubs, share, seed):
    """A random game where a share of the edges goes to a few vertices; edges
    may repeat and loop."""
    r = np.random.default_rng(seed)
    deg = r.integers(1, 6, n)
    off = np.zeros(n + 1, np.int32)
    np.cumsum(deg, out=off[1:])
    m = int(off[-1])
    tgt = np.where(r.random(m) < share, r.integers(0, hubs, m) * (n // hubs), r.integers(0, n, m)).astype(np.int32)
    return Game(n, off, tgt, (r.random(n) < 0.5).astype(np.uint8), r.permutation(n).astype(np.int32))


def check(pg, ctx, g, reset=False):
    _, res, want = o2.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri, reset=reset)
    game = pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    try:
        out = dict(win=np.empty(g.n, np.uint8), val_class=np.empty(g.n, np.int8),
                   **{k: np.empty(g.n, np.int32) for k in ("sigma", "tau", "val_depth", "val_rank")})
        for _ in range(2):  # the second solve starts from the first one's marks and lists
            got = pg.pg_solve(ctx, game, reset_tau=reset, **out)
            assert got == (want["major"], want["inner"])
            for k in KEYS:
                assert np.array_equal(out[k], np.asarray(want[k])), k
    finally:
        pg.pg_game_free(game)


@pytest.mark.parametrize("n", [1, 2, 33, 900, 1023, 1024, 1025, 2100, 16383, 16385, 45000, 70001, 130000])
@pytest.mark.parametrize("shape", ["random", "ladder"])
def test_sizes(pg, ctx, shape, n):
    check(pg, ctx, gen.ladder_game(max(n, 2), n) if shape == "ladder" else gen.native_random_game(n, 1, 6, seed=n))


@pytest.mark.parametrize("n,hubs,share", [(3000, 1, 0.4), (20000, 3, 0.5), (20000, 12, 0.1), (90000, 2, 0.3),
                                          (90000, 60, 0.3), (150000, 9, 0.02)])
def test_many_predecessors(pg, ctx, n, hubs, share):
    check(pg, ctx, hub_game(n, hubs, share, n + hubs))


@pytest.mark.parametrize("n", [700, 30000, 100003])
def test_reset(pg, ctx, n):
    check(pg, ctx, gen.native_random_game(n, 2, 5, seed=n), reset=True)


@pytest.mark.parametrize("levels", [2, 4])
@pytest.mark.parametrize("n,hubs,share", [(900, 1, 0.0), (20000, 3, 0.3), (150001, 50, 0.0), (150001, 4000, 0.4)])
def test_few_priorities(pg, ctx, n, hubs, share, levels):
    g = hub_game(n, hubs, share, n + hubs)
    g.pri[:] = g.pri % levels
    _, _, want = o3.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)
    game = pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    try:
        d = pg.pg_game_levels(game).size
        out = dict(win=np.empty(n, np.uint8), val_class=np.empty(n, np.int8), val_counts=np.empty(n * d, np.int32),
                   **{k: np.empty(n, np.int32) for k in ("sigma", "tau", "val_depth")})
        for _ in range(2):
            assert pg.pg_solve(ctx, game, **out) == (want["major"], want["inner"])
            for k in out:
                assert np.array_equal(out[k].reshape(np.asarray(want[k]).shape), np.asarray(want[k])), k
    finally:
        pg.pg_game_free(game)
