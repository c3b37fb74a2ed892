"""Loads of games with sparse priorities: in one launch while the priority
bitmap is small enough, by the general path beyond, with odd and even
priorities among them."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1705_02313_gb300 import gen
from paper_1705_02313_gb300.gen import Game

from test_gpu_parity import assert_same, oracle_solution

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


def sparse(n, top, seed):
    """Distinct random priorities up to top (which occurs), of both parities."""
    g = gen.native_random_game(n, 1, 5, seed=seed)
    rng = np.random.default_rng(seed)
    pri = rng.permutation(n).astype(np.int64) * max(top // n, 1)
    if top >= 2 * n:
        pri += rng.integers(0, top // n, n)
        pri[np.argmax(pri)] = top
    assert np.unique(pri).size == n and set(pri % 2) == {0, 1}
    return Game(n, g.offsets, g.targets, g.owner, pri.astype(np.int32))


def load_launches(pg, ctx, g, device):
    arrays = [torch.from_numpy(x).cuda() for x in g.arrays()] if device else g.arrays()
    l0 = launches(pg, ctx)
    game = pg.pg_load_csr(ctx, g.n, g.m, *arrays)
    took = launches(pg, ctx) - l0
    pg.pg_game_free(game)
    return took


# the bitmap of n vertices has max(2 n + 2048, min(2^21, 64 n)) words, and priorities are raised by up to 2 n
@pytest.mark.parametrize("n", [40, 1000, 20_000, 30_000, 40_000])
def test_up_to_the_bitmap(pg, ctx, n):
    words = max(2 * n + 2048, min(1 << 21, 64 * n))
    fits = 32 * words - 2 * n - 1
    for top, one in ((3 * n, True), (fits, True), (fits + 1, False), (min(40 * fits, 2**31 - 1 - 2 * n), False)):
        g = sparse(n, top, n)
        for device in (False, True):
            assert (load_launches(pg, ctx, g, device) == 1) == one, (n, top, device)
        assert_same(pg.solve_arrays(ctx, g.n, *g.arrays()), oracle_solution(g)[2], "n=%d top=%d" % (n, top))


def test_sparse_host_arrays_are_not_tried(pg, ctx):
    """The first priorities of host arrays tell; those of device arrays take a launch."""
    g = sparse(300_000, 2**30, 5)
    assert load_launches(pg, ctx, g, False) == load_launches(pg, ctx, g, True) - 1


@pytest.mark.parametrize("wide", [0, 1])
@pytest.mark.parametrize("spread", [1, 7, 100, 3000])
def test_batches(pg, ctx, spread, wide):
    """One union while the priorities are dense enough, game by game beyond; odd and even priorities in all."""
    from test_gpu_batch import KEYS, run_batch
    pg.pg_set_wide_offsets(ctx, wide)
    games = [sparse(n, n * spread, n) for n in (900, 60, 5000, 2500)]
    vb, res, out = run_batch(pg, ctx, games)
    assert res["rc"] == pg.PG_OK
    for i, g in enumerate(games):
        want = oracle_solution(g)[2]
        for k in KEYS:
            assert np.array_equal(out[k][int(vb[i]):int(vb[i + 1])], np.asarray(want[k])), (i, k)
