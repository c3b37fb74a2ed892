"""Several threads, each with its own context and stream, load, solve and free
games of a size whose loops are captured as graphs: freeing waits for the
device, which must not happen while another thread captures. In a process of
its own (a dropped capture has crashed it). Results are those of one thread."""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
THREADS, ROUNDS, N = 8, 8, 90_000


def test_threads():
    from paper_1705_02313_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-3000:]


def main():
    sys.path.insert(0, os.path.dirname(HERE))
    import torch

    from paper_1705_02313_gb300 import gen, pg
    torch.zeros(1, device="cuda")
    games = [gen.native_random_game(N, 2, 6, seed=i) for i in range(THREADS)]
    failed, results = [], [[] for _ in games]

    def run(i, rounds):
        g = games[i]
        try:
            ctx = pg.pg_ctx_create(0)
            pg.pg_set_stream(ctx, torch.cuda.Stream())
            for _ in range(rounds):
                out = dict(win=np.empty(N, np.uint8), sigma=np.empty(N, np.int32), val_rank=np.empty(N, np.int32))
                game = pg.pg_load_csr(ctx, N, g.m, *g.arrays())
                counts = pg.pg_solve(ctx, game, **out)
                pg.pg_game_free(game)
                results[i].append((counts, out))
            pg.pg_ctx_destroy(ctx)
        except Exception as e:  # reported below
            failed.append((i, repr(e)))

    for i in range(THREADS):
        run(i, 1)
    threads = [threading.Thread(target=run, args=(i, ROUNDS)) for i in range(THREADS)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    for r in results:
        assert len(r) == ROUNDS + 1
        for counts, out in r[1:]:
            assert counts == r[0][0]
            for k in out:
                assert np.array_equal(out[k], r[0][1][k]), k


if __name__ == "__main__":
    main()
