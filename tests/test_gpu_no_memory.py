"""Allocations that fail (alloc_shim.cpp, in a process of its own): each one of
a call in turn. What the library can do without costs time only: a game is
loaded the general way, a batch game by game, loops run without the reverse
lists. Results stay the oracle's, an error leaves the handle usable, and
nothing else is returned than PG_ENOMEM."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CASES = ["load", "load_all", "solve_whole", "solve_graph", "solve_levels", "solve_deep", "batch"]


@pytest.mark.parametrize("case", CASES)
def test_failing_allocations(case, tmp_path):
    from paper_1705_02313_gb300 import build
    build.build()
    shim = str(tmp_path / "shim.so")
    r = subprocess.run(["g++", "-O1", "-fPIC", "-shared", os.path.join(HERE, "alloc_shim.cpp"), "-o", shim, "-ldl"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    env = dict(os.environ, SHIM=shim, SHIM_LIBPG=build.LIB)
    r = subprocess.run([sys.executable, os.path.abspath(__file__), case], capture_output=True, text=True, env=env,
                       timeout=300)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]


# ---------------------------------------------------------------------------
# the child

def arrays_of(n):
    return dict(win=np.full(n, 77, np.uint8), sigma=np.full(n, 77, np.int32), tau=np.full(n, 77, np.int32),
                val_class=np.full(n, 77, np.int8), val_depth=np.full(n, 77, np.int32))


class Child:
    def __init__(self):
        import ctypes
        self.shim = ctypes.CDLL(os.environ["SHIM"], mode=ctypes.RTLD_GLOBAL)
        self.shim.shim_fail.argtypes = [ctypes.c_long, ctypes.c_long]
        self.shim.shim_calls.restype = ctypes.c_long
        sys.path[:0] = [os.path.dirname(HERE), HERE]
        from paper_1705_02313_gb300 import pg
        self.pg = pg
        self.ctx = pg.pg_ctx_create(0, tuning=False)
        self.load(self.random(50, 1), free=True)
        assert self.shim.shim_calls() > 0, "the shim is not in use"

    def random(self, n, seed, **kw):
        from paper_1705_02313_gb300 import gen
        return gen.native_random_game(n, 1, 5, seed=seed, **kw)

    def load(self, g, free=False):
        game = self.pg.pg_load_csr(self.ctx, g.n, g.m, *g.arrays())
        if free:
            self.pg.pg_game_free(game)
        return game

    def want(self, g):
        from oracle import o2, o3
        solver = o2 if np.unique(g.pri).size == g.n else o3
        return solver.solve_game(g.n, g.offsets, g.targets, g.owner, g.pri)[2]

    def solved(self, game, g, want):
        out = arrays_of(g.n)
        got = self.pg.pg_solve(self.ctx, game, **out)
        assert got == (want["major"], want["inner"])
        for key in out:
            assert np.array_equal(out[key], np.asarray(want[key])), key

    def each_failing(self, call, after, count=1):
        """Runs call with its 1st, 2nd, ... allocation failing (and the count - 1 after it) until none does, after
        each time without failures; the numbers that gave PG_ENOMEM."""
        refused = []
        for k in range(400):
            self.shim.shim_fail(k, count)
            got = None
            try:
                got = call()
            except self.pg.PgError as e:
                assert e.code == self.pg.PG_ENOMEM, (k, str(e))
                refused.append(k)
            made = self.shim.shim_calls()
            self.shim.shim_fail(-1, 0)
            after(got)
            if made <= k:
                return refused
        raise AssertionError("more allocations than expected")

    def load_case(self, all_from):
        """One allocation fails: the general path loads. All from one on: refused."""
        for n in (3000, 30_000):
            g = self.random(n, n)
            want = self.want(g)

            def after(game):
                game = game or self.load(g)
                self.solved(game, g, want)
                self.pg.pg_game_free(game)

            refused = self.each_failing(lambda: self.load(g), after, 1000 if all_from else 1)
            assert bool(refused) == all_from, refused

    def solve_case(self, g, needed):
        """needed: the allocations that a solve cannot do without. The handle stays usable, with lists or without."""
        want = self.want(g)
        games = [self.load(g)]

        def after(_):
            for _ in range(2):
                self.solved(games[0], g, want)
            self.pg.pg_game_free(games[0])
            games[0] = self.load(g)

        refused = self.each_failing(lambda: self.solved(games[0], g, want), after)
        assert len(refused) == needed, refused

    def batch_case(self):
        """Only the batch's own scratch is needed."""
        import test_gpu_batch as tb
        games = [self.random(n, n) for n in (400, 1500, 900)]
        wants = [self.want(g) for g in games]

        def check(ran):
            vb, res, out = ran or tb.run_batch(self.pg, self.ctx, games)
            assert res["rc"] == self.pg.PG_OK
            for i, want in enumerate(wants):
                sl = slice(int(vb[i]), int(vb[i + 1]))
                for key in ("win", "sigma", "tau", "val_class", "val_depth", "val_rank"):
                    assert np.array_equal(out[key][sl], np.asarray(want[key])), (i, key)

        refused = self.each_failing(lambda: tb.run_batch(self.pg, self.ctx, games), check)
        assert len(refused) == 1, refused


def main(case):
    c = Child()
    if case == "load":
        c.load_case(False)
    elif case == "load_all":
        c.load_case(True)
    elif case == "solve_whole":
        c.solve_case(c.random(3000, 5), 0)
    elif case == "solve_graph":
        c.solve_case(c.random(90_000, 6), 6)  # the players' views
    elif case == "solve_levels":
        c.solve_case(c.random(70_000, 7, levels=4), 0)
    elif case == "solve_deep":
        from test_gpu_deep import climbing_game
        c.solve_case(climbing_game(3000, 3, 0.05), 0)
    elif case == "batch":
        c.batch_case()
    c.pg.pg_ctx_destroy(c.ctx)


if __name__ == "__main__":
    main(sys.argv[1])
