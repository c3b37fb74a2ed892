"""Count-vector solves that end with incremental iterations: the outputs that
the keys alone give (no depths), Even's passes over all ids inside the
incremental launch (games of up to 65,536 ids) and outside it, against the
oracle and against a call that asks for everything."""
import ctypes as C

import numpy as np
import pytest

from oracle import o3
from paper_1705_02313_gb300 import gen

pytestmark = pytest.mark.gpu

KEYS = ["win", "sigma", "tau", "val_class", "val_counts"]


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


@pytest.mark.parametrize("n", [2, 40, 1000, 1600, 4096, 26000, 48000, 56000, 90000])
@pytest.mark.parametrize("shape", ["random", "ladder"])
def test_outputs_from_the_keys(pg, ctx, shape, n):
    g = gen.ladder_game(n, n) if shape == "ladder" else gen.native_random_game(n, 1, 5, seed=n, levels=4)
    if shape == "ladder":
        g.pri[:] = g.pri % 3
    if np.unique(g.pri).size == n:  # (tiny games may draw distinct priorities)
        pytest.skip("distinct priorities")
    _, _, want = o3.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)
    game = pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    try:
        d = pg.pg_game_levels(game).size
        out = dict(win=np.empty(n, np.uint8), sigma=np.empty(n, np.int32), tau=np.empty(n, np.int32),
                   val_class=np.empty(n, np.int8), val_counts=np.empty(n * d, np.int32))
        depth = np.empty(n, np.int32)
        took = []
        for more in (dict(val_depth=depth), {}, dict(val_depth=depth), {}):
            for x in out.values():
                x.fill(77)
            l0 = launches(pg, ctx)
            assert pg.pg_solve(ctx, game, **out, **more) == (want["major"], want["inner"])
            took.append(launches(pg, ctx) - l0)
            for k in KEYS:
                assert np.array_equal(out[k].reshape(np.asarray(want[k]).shape), np.asarray(want[k])), (k, more.keys())
            if more:
                assert np.array_equal(depth, np.asarray(want["val_depth"]))
            assert pg.pg_game_counters(game)["n_fin"] >= int((np.asarray(want["val_class"]) == 0).sum())
        # a full valuation (four kernels) and the depth pass against one kernel, where the loop ended incrementally
        if n >= 1000:
            assert took[2] - took[3] == 4, took
        tau = np.full(n, 77, np.int32)
        val = np.full(n, 77, np.int8)
        _, _, k = pg.pg_game_info(game)
        dsig = np.empty(max(k, 1), np.int8)
        pg.pg_solve(ctx, game, sigma=out["sigma"], dummy_sigma=dsig)
        counts = np.full(n * d, 77, np.int32)
        pg.pg_best_response(ctx, game, out["sigma"], dummy_sigma=dsig[:k] if k else None, val_class=val,
                            val_counts=counts)
        assert np.array_equal(val, np.asarray(want["val_class"]))
        assert np.array_equal(counts.reshape(n, d), np.asarray(want["val_counts"]))
    finally:
        pg.pg_game_free(game)
