"""Incremental iterations at the ends of their lists (csrc/pg_inc.cu): queues of
Odd's and Even's vertices beyond what a block holds, for a game solved in one
launch, for one solved by the loop graph and for packed ones, and count-vector
plays longer inside the affected set than a key is summed over. All against
the oracle."""
import numpy as np
import pytest

from oracle import o3
from paper_1705_02313_gb300.gen import Game

from test_gpu_batch import KEYS, run_batch
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


class Maker:
    """Vertices in increasing order of priority: owner, parity, successors."""

    def __init__(self):
        self.rows, self.own, self.odd = [], [], []

    def add(self, own, odd, succ=()):
        self.rows.append(list(succ))
        self.own.append(own)
        self.odd.append(odd)
        return len(self.rows) - 1

    def loops(self, count, odd=0):
        """Even's vertices with a self-loop: they go to the sink."""
        out = [self.add(0, odd) for _ in range(count)]
        for v in out:
            self.rows[v] = [v]
        return out

    def game(self, seed):
        n = len(self.rows)
        at = np.random.default_rng(seed).permutation(n)  # vertex ids in any order
        rows = [None] * n
        own, pri = np.empty(n, np.uint8), np.empty(n, np.int32)
        for v in range(n):
            rows[at[v]] = [int(at[x]) for x in self.rows[v]]
            own[at[v]] = self.own[v]
            pri[at[v]] = 2 * v + self.odd[v]
        off = np.zeros(n + 1, np.int32)
        off[1:] = np.cumsum([len(r) for r in rows])
        return Game(n, off, np.array([x for r in rows for x in r], np.int32), own, pri)


def odd_queue_game(hubs, each, fill, steps=4, seed=1):
    """One Odd vertex after the other switches (a staircase of steps vertices);
    the last one changes the top of hubs vertices that each have `each` Odd
    predecessors, which stay where they are."""
    m = Maker()
    m.loops(fill)
    ends = m.loops(8)
    low = m.loops(steps)
    # Odd's vertices behind the hubs: their first choice is better for Odd than what the hubs come to
    last = m.add(1, 0)
    stairs = [m.add(1, 0) for _ in range(steps - 1)] + [last]
    hub = [m.add(1, 0, [last]) for _ in range(hubs)]
    w = m.add(0, 1)  # the large odd priority at the foot of the stairs
    m.rows[w] = [w]
    best = m.add(0, 1)
    m.rows[best] = [best]
    for k, d in enumerate(stairs):
        m.rows[d] = [low[k], w if k == 0 else stairs[k - 1]]
    for h in hub:
        for _ in range(each):
            m.add(1, 0, [best, h])
    assert ends
    return m.game(seed)


def even_queue_game(hubs, each, fill, seed=2):
    """Even's first pass switches one vertex; what it leads to then makes the
    hubs better than the sink for `each` Even predecessors of each of them."""
    m = Maker()
    m.loops(fill)
    behind = [[m.add(0, 0) for _ in range(each)] for _ in range(hubs)]
    e = m.add(0, 0)
    hub = [m.add(1, 1, [e]) for _ in range(hubs)]
    y = m.add(0, 0)
    m.rows[y] = [y]
    m.rows[e] = [y]
    for h, row in zip(hub, behind):
        for v in row:
            m.rows[v] = [h]
    return m.game(seed)


def want_of(g):
    return oracle_solution(g)[2]


@pytest.mark.parametrize("hubs,each,fill", [(24, 1000, 0), (40, 1024, 2000), (24, 1000, 60_000), (3, 1025, 90_000)])
def test_odd_queue(pg, ctx, hubs, each, fill):
    g = odd_queue_game(hubs, each, fill)
    assert_same(pg.solve_arrays(ctx, g.n, *g.arrays()), want_of(g), "odd queue")


@pytest.mark.parametrize("hubs,each,fill", [(18, 1000, 0), (40, 1024, 1000), (20, 1000, 60_000)])
def test_even_queue(pg, ctx, hubs, each, fill):
    g = even_queue_game(hubs, each, fill)
    want = want_of(g)
    assert want["major"] >= 2
    assert_same(pg.solve_arrays(ctx, g.n, *g.arrays()), want, "even queue")


@pytest.mark.parametrize("copies", [3, 200])
def test_queues_of_packed_games(pg, ctx, copies):
    """3 games: one or several blocks of 1,024 threads each; 200: blocks of a quarter of them."""
    small = copies > 100
    games = [odd_queue_game(3, 1000, 100, seed=i) if small else odd_queue_game(10, 1000, 100, seed=i)
             for i in range(copies // 2)]
    games += [even_queue_game(5, 1000, 0, seed=i) if small else even_queue_game(18, 1000, 0, seed=i)
              for i in range(copies - len(games))]
    wants = [want_of(g) for g in games]
    vb, res, out = run_batch(pg, ctx, games)
    assert res["rc"] == pg.PG_OK
    for i, want in enumerate(wants):
        sl = slice(int(vb[i]), int(vb[i + 1]))
        for k in KEYS:
            assert np.array_equal(out[k][sl], np.asarray(want[k])), (i, k)


@pytest.mark.parametrize("segments,length,fill", [(15, 24, 6000), (9, 20, 6000), (60, 24, 30_000)])
def test_long_keys(pg, ctx, segments, length, fill):
    """A play through segments that each end in a choice between an even and an
    odd priority: Odd switches all of them at once, and the keys of the play
    run through every segment (count vectors, 15 x 24 vertices: beyond the 256
    that a key is summed over)."""
    rows, own, pri = [], [], []

    def add(o, p, succ):
        rows.append(succ)
        own.append(o)
        pri.append(p)
        return len(rows) - 1

    nxt = add(0, 2, [])
    rows[nxt] = [nxt]
    rng = np.random.default_rng(segments)
    for _ in range(segments):
        u, v = add(1, 2, [nxt]), add(1, 3, [nxt])
        nxt = add(1, int(rng.integers(0, 2)), [u, v])
        for _ in range(length):
            nxt = add(1, int(rng.integers(0, 2)), [nxt])
    for _ in range(fill):
        v = add(0, int(rng.integers(0, 4)), [])
        rows[v] = [v]
    n = len(rows)
    off = np.zeros(n + 1, np.int32)
    off[1:] = np.cumsum([len(r) for r in rows])
    g = Game(n, off, np.array([x for r in rows for x in r], np.int32), np.array(own, np.uint8),
             np.array(pri, np.int32))
    want = o3.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)[2]
    game = pg.pg_load_csr(ctx, n, g.m, *g.arrays())
    try:
        d = pg.pg_game_levels(game).size
        out = dict(win=np.empty(n, np.uint8), sigma=np.empty(n, np.int32), tau=np.empty(n, np.int32),
                   val_class=np.empty(n, np.int8), val_depth=np.empty(n, np.int32),
                   val_counts=np.empty(n * d, np.int32))
        for _ in range(2):
            assert pg.pg_solve(ctx, game, **out) == (want["major"], want["inner"])
            for k in out:
                assert np.array_equal(out[k].reshape(np.asarray(want[k]).shape), np.asarray(want[k])), k
    finally:
        pg.pg_game_free(game)
