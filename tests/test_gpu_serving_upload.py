"""Submitted databases on their way to the device: uploaded through pinned buffers while the budget has room, copied on the host
behind a job that waits for room or with offsets that the build refuses; the caller's arrays are free after the call."""
import threading
import time

import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import fim, synth

pytestmark = pytest.mark.gpu


def odict(res):
    so, si, sp = res
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


def requests(n):
    return [(*synth.request_db(r), r["N"], max(2, r["minsup"]))
            for r in synth.serving_requests(n, seed=5, D_range=(500, 8_000), N_range=(20, 300), TL_range=(4.0, 9.0),
                                            rel_range=(0.01, 0.05))]


# every job's footprint is 64 MB and a little more: none, one at a time, or all uploaded
@pytest.mark.parametrize("budget", [1, 100 << 20, 0])
def test_results_with_arrays_reused_after_submit(budget):
    reqs = requests(6)
    srv = fim.Server(hbm_budget_bytes=budget, slots=3)
    try:
        ids = []
        for off, items, N, ms in reqs:
            o, i = off.copy(), items.copy()
            ids.append(srv.submit(o, i, N, ms, sample_rate=0.2))
            o[:] = 0
            i[:] = N + 1
        for jid, (off, items, N, ms) in zip(ids, reqs):
            assert srv.wait(jid)[0].as_dict() == odict(oracle.eclat(off, items, N, ms))
        st = srv.stats()
        assert st["in_use_bytes"] == 0 and st["queued"] == 0 and st["in_flight"] == 0
        assert st["peak_in_flight"] == 1 or budget == 0
    finally:
        srv.free()


@pytest.mark.parametrize("D,per", [(1, 1), (65_537, 1), (400_001, 13), (2_500_000, 7)])
def test_databases_of_several_pieces(D, per):
    """Uploads of one piece and of many, of sizes that end within one: the same counts as a database built directly."""
    rng = np.random.default_rng(D)
    off = (np.arange(D + 1) * per).astype(np.uint32)
    items = (rng.integers(0, 30, size=(D, per)) + 30 * np.arange(per)).astype(np.uint32).reshape(-1)
    N, minsup = 30 * per, max(1, D // 1_000)
    db = fim.build_vertical_db(off, items, N)
    want = db.mine(minsup).as_dict()
    db.free()
    srv = fim.Server(slots=2)
    try:
        ids = [srv.submit(off.copy(), items.copy(), N, minsup) for _ in range(3)]
        for jid in ids:
            assert srv.wait(jid)[0].as_dict() == want
    finally:
        srv.free()


def test_a_long_copy_holds_up_no_other_job():
    """While one thread's large database is copied on the host (no budget for an upload), another's small job, submitted
    after it, is mined and returned."""
    D, per = 15_000_000, 20
    off = (np.arange(D + 1, dtype=np.int64) * per).astype(np.uint32)
    items = (np.arange(D * per, dtype=np.uint32)) % 1_000
    small = requests(1)[0]
    want = odict(oracle.eclat(*small))
    srv = fim.Server(hbm_budget_bytes=1, slots=2)
    try:
        srv.wait(srv.submit(*small))  # (the first job of a server allocates)
        big = {}

        def submit_big():
            big["id"] = srv.submit(off, items, 1_000, D)  # (no frequent item)
            big["submitted"] = time.perf_counter()

        t = threading.Thread(target=submit_big)
        t.start()
        while srv.stats()["queued"] == 0 and t.is_alive():
            time.sleep(0.0005)
        res = srv.wait(srv.submit(*small))[0]
        done = time.perf_counter()
        assert res.as_dict() == want
        t.join()
        assert done < big["submitted"]
        assert srv.wait(big["id"])[0].n_sets == 0
        assert srv.stats()["in_use_bytes"] == 0
    finally:
        srv.free()


def test_refused_and_empty_databases():
    srv = fim.Server(slots=2)
    try:
        items = np.zeros(4, dtype=np.uint32)
        for off in ([1, 2, 4], [0, 3, 2, 4]):  # does not start at 0; decreases
            jid = srv.submit(np.array(off, dtype=np.uint32), items, 3, 1)
            with pytest.raises(fim.FimError) as e:
                srv.wait(jid)
            assert e.value.status == fim.FIM_ERR_INVALID and "tx_offsets" in str(e.value)
        assert srv.wait(srv.submit(np.zeros(9, dtype=np.uint32), items[:0], 3, 1))[0].n_sets == 0
        assert srv.stats()["in_use_bytes"] == 0
    finally:
        srv.free()


def test_freed_with_jobs_queued():
    srv = fim.Server(slots=1)
    for off, items, N, ms in requests(4):
        srv.submit(off, items, N, ms)
    srv.free()
