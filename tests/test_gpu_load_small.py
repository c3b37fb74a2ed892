"""Games loaded in one launch (csrc/pg_load_small.cu): its dummies and solutions
around the sizes of a block, the cluster and the grid, and the games that it
hands to the general path."""
import numpy as np
import pytest

from oracle import o2
from paper_1705_02313_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    from paper_1705_02313_gb300 import pg
    return pg


@pytest.fixture(scope="module")
def ctx(pg):
    c = pg.pg_ctx_create(0)
    yield c
    pg.pg_ctx_destroy(c)


def check(pg, ctx, g, device=False):
    import torch
    gp = o2.preprocess(g.n, *g.arrays())
    want = o2.map_back(gp, o2.run(gp))
    arrays = [torch.from_numpy(a).cuda() for a in g.arrays()] if device else g.arrays()
    game = pg.pg_load_csr(ctx, g.n, g.m, *arrays)
    try:
        assert pg.pg_game_info(game) == (g.n, g.m, gp["k"])
        assert np.array_equal(pg.pg_game_dummies(game), gp["dummy_of"])
        out = dict(win=np.empty(g.n, np.uint8), sigma=np.empty(g.n, np.int32), tau=np.empty(g.n, np.int32),
                   val_rank=np.empty(g.n, np.int32))
        pg.pg_solve(ctx, game, **out)
    finally:
        pg.pg_game_free(game)
    for k in out:
        assert np.array_equal(out[k], np.asarray(want[k])), k


@pytest.mark.parametrize("n", [1, 2, 1023, 1025, 8191, 24576, 24577, 90001])
@pytest.mark.parametrize("shape", ["random", "ladder", "odd"])
def test_sizes(pg, ctx, n, shape):
    if shape == "ladder":
        g = gen.ladder_game(max(n, 2), n, p_odd=0.9)
    else:
        g = gen.native_random_game(n, 1, 4, seed=n, p_odd=0.5 if shape == "random" else 1.0)
    check(pg, ctx, g, device=n % 2 == 1)


def test_sparse_and_repeated_priorities(pg, ctx):
    g = gen.random_game(3000, 1, 4, 5)
    g.pri[:] = g.pri * 600_000  # beyond the kernel's bitmap
    check(pg, ctx, g)
    g = gen.random_game(3000, 1, 4, 6)
    g.pri[np.argmax(g.pri)] = np.sort(g.pri)[-2]  # one repeat, not among the first vertices
    with pytest.raises(pg.PgError) as e:
        pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    assert e.value.code == pg.PG_EUNSUPPORTED
    g = gen.random_game(3000, 1, 4, 7)
    g.targets[1234] = 3000
    with pytest.raises(pg.PgError) as e:
        pg.pg_load_csr(ctx, g.n, g.m, *g.arrays())
    assert e.value.code == pg.PG_EINVAL and "target" in str(e.value)
