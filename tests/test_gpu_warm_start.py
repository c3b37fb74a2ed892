"""Solves from a given strategy on a game just loaded: the first iterations run
without views, lists or a graph, the rest with them. From the solution (two
iterations), from a profile on the way to it (more than those first ones), with
few priorities and with distinct ones, shallow and deep, against the same solve
without graphs; and what a solve that ends at once does not launch."""
import ctypes as C

import numpy as np
import pytest

from paper_1705_02313_gb300 import gen

from test_gpu_deep import climbing_game

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


def launches(pg, ctx):
    x = C.c_int64()
    pg.lib().pg_launch_count(ctx, C.byref(x))
    return x.value


def outputs(n, k):
    return dict(win=np.full(n, 77, np.uint8), sigma=np.full(n, 77, np.int32), tau=np.full(n, 77, np.int32),
                val_class=np.full(n, 77, np.int8), val_depth=np.full(n, 77, np.int32),
                val_rank=np.full(n, 77, np.int32), dummy_sigma=np.full(max(k, 1), 77, np.int8))


def solve(pg, ctx, g, start=None, cap=0, again=False):
    """(counts, outputs, launches) of a solve on a fresh handle."""
    game = pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    try:
        out = outputs(g.n, pg.pg_game_info(game)[2])
        for _ in range(2 if again else 1):
            l0 = launches(pg, ctx)
            try:
                counts = pg.pg_solve(ctx, game, **out, max_inner=cap,
                                     **({} if start is None else dict(sigma_init=start["sigma"], tau_init=start["tau"],
                                                                      dummy_sigma_init=start["dummy_sigma"])))
            except pg.PgError as e:
                assert e.code == pg.PG_ETIMEOUT and cap
                counts = None
            took = launches(pg, ctx) - l0
    finally:
        pg.pg_game_free(game)
    return counts, out, took


GAMES = {
    "random": lambda: gen.native_random_game(90_000, 1, 5, seed=1),
    "ladder": lambda: gen.ladder_game(120_000, 2),
    "levels": lambda: gen.native_random_game(70_000, 1, 5, seed=3, levels=4),
    "small levels": lambda: gen.native_random_game(3_000, 2, 5, seed=4, levels=3),
    "deep": lambda: climbing_game(80_000, 5, 0.02),
}


@pytest.mark.parametrize("name", sorted(GAMES))
@pytest.mark.parametrize("cap", [0, 1, 4, 15])
def test_warm_starts(pg, ctx, name, cap):
    """cap: the start is where a cold solve stands after that many iterations (0: the solution)."""
    g = GAMES[name]()
    _, start, _ = solve(pg, ctx, g, cap=cap)
    pg.pg_set_graphs(ctx, 0)
    counts, want, _ = solve(pg, ctx, g, start)
    pg.pg_set_graphs(ctx, 1)
    for again in (False, True):
        got, out, _ = solve(pg, ctx, g, start, again=again)
        assert got == counts
        for k in want:
            assert np.array_equal(out[k], want[k]), (k, again)
    # a cap inside the first iterations, and one at their end
    for limit in (1, 2, 3):
        pg.pg_set_graphs(ctx, 0)
        a = solve(pg, ctx, g, start, cap=limit)
        pg.pg_set_graphs(ctx, 1)
        b = solve(pg, ctx, g, start, cap=limit)
        assert a[0] == b[0]
        for k in a[1]:
            assert np.array_equal(a[1][k], b[1][k]), (k, limit)


@pytest.mark.parametrize("name", ["random", "levels"])
def test_a_solution_that_holds_needs_no_lists(pg, ctx, name):
    g = GAMES[name]()
    _, start, _ = solve(pg, ctx, g)
    counts, _, took = solve(pg, ctx, g, start)
    pg.pg_set_graphs(ctx, 0)  # (no incremental iterations, so no lists for them; views for distinct priorities)
    assert solve(pg, ctx, g, start)[0] == counts
    bare = solve(pg, ctx, g, start)[2]
    assert took <= bare - (10 if name == "random" else 0), (took, bare)
