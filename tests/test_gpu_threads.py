"""Databases of several threads, each on a stream of its own (GPU): a short mine does not wait for the end of another
thread's long one, whichever kernels it takes, and the results are those of the mines alone."""
import threading
import time

import numpy as np
import pytest

from paper_2108_05038_gb300 import fim, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def long_mine():
    """A database whose mine in sparse nodes holds every SM for tens of milliseconds."""
    D, N = 500_000, 8_000
    off, items = synth.pattern_db(5, D, N, 20.0, 6.0, 2 * N, "zipf")
    return off, items, N, synth.abs_minsup(0.0006, D)


# by levels (fewer than 1,024 rows); small subtrees in shared memory (the projected mode's)
@pytest.mark.parametrize("D,N,rel,mode", [(10_000, 100, 0.01, None), (30_000, 300, 0.005, fim.FIM_DFS_PROJECTED)])
def test_short_mines_beside_a_long_one(long_mine, D, N, rel, mode):
    import torch

    off, items = synth.pattern_db(3, D, N, 10.0, 4.0, 2 * N, "uniform")
    minsup = synth.abs_minsup(rel, D)
    want = None
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    big = fim.build_vertical_db(*long_mine[:3], stream=streams[0])
    db = fim.build_vertical_db(off, items, N, stream=streams[1])
    kw = dict(stats=False) if mode is None else dict(stats=False, dfs_mode=mode)
    try:
        want = db.mine(minsup, **kw).as_dict()
        stop, long_ms, failed = threading.Event(), [], []

        def run_long():
            try:
                while not stop.is_set():
                    t = time.perf_counter()
                    big.mine(long_mine[3], dfs_mode=fim.FIM_DFS_SPARSE, result_on_device=True, stats=False).free()
                    long_ms.append((time.perf_counter() - t) * 1e3)
            except Exception as e:  # (reported by the test's thread)
                failed.append(e)

        big.mine(long_mine[3], dfs_mode=fim.FIM_DFS_SPARSE, result_on_device=True, stats=False).free()
        t = threading.Thread(target=run_long)
        t.start()
        short_ms = []
        try:
            end = time.perf_counter() + 1.0
            while time.perf_counter() < end:
                t0 = time.perf_counter()
                got = db.mine(minsup, **kw)
                short_ms.append((time.perf_counter() - t0) * 1e3)
                assert got.n_sets == len(want)
                last = got
        finally:
            stop.set()
            t.join()
        assert not failed
        assert last.as_dict() == want
        # (the long mine's CTAs leave one by one at its end, and a waiting launch that needs all SMs at once starts only
        # then: its median is the long mine's length)
        assert np.median(short_ms) < 0.25 * np.median(long_ms), (np.median(short_ms), np.median(long_ms))
    finally:
        big.free()
        db.free()
