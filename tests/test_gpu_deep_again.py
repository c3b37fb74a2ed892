"""Games that turn deep, solved more than once on the same handle: the second
solve replays the loop graph of the first, whose ruling-set valuations write the
depths and are reported as deep like the first's."""
import ctypes as C

import numpy as np
import pytest

from test_gpu_deep import climbing_game
from test_gpu_parity import oracle_solution

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


@pytest.mark.parametrize("n,back,seed", [(3000, 0.0, 1), (4000, 0.1, 5)])
@pytest.mark.parametrize("ranks", [0, 1])
def test_solved_again(pg, ctx, n, back, seed, ranks):
    g = climbing_game(n, seed, back)
    _, _, want = oracle_solution(g)
    pg.pg_set_loop_ranks(ctx, ranks)
    game = pg.pg_load_csr(ctx, n, g.m, *g.arrays())
    try:
        out = dict(win=np.empty(n, np.uint8), sigma=np.empty(n, np.int32), tau=np.empty(n, np.int32),
                   val_class=np.empty(n, np.int8), val_rank=np.empty(n, np.int32))
        depth = np.empty(n, np.int32)
        took = []
        for more in (dict(val_depth=depth), dict(val_depth=depth), {}, dict(val_depth=depth)):
            depth.fill(77)
            l0 = launches(pg, ctx)
            assert pg.pg_solve(ctx, game, **out, **more) == (want["major"], want["inner"])
            took.append(launches(pg, ctx) - l0)
            assert pg.pg_game_counters(game)["deep"] == 1
            for k in out:
                assert np.array_equal(out[k], np.asarray(want[k])), k
            if more:
                assert np.array_equal(depth, np.asarray(want["val_depth"]))
        if not ranks:  # the ruling-set path wrote the depths: no pass of its own for them
            assert took[1] == took[2] == took[3], took
        # a shallow valuation in between
        pg.pg_valuate(ctx, game, np.full(n, -1, np.int32), None, None, val_depth=depth)
        pg.pg_solve(ctx, game, **out, val_depth=depth)
        assert pg.pg_game_counters(game)["deep"] == 1
        assert np.array_equal(depth, np.asarray(want["val_depth"]))
    finally:
        pg.pg_game_free(game)
