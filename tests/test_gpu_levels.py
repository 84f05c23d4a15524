"""The search by levels (GPU; the automatic traversal of mines of fewer than 1,024 rows) against the frame passes (the same
nodes, intersections and class work) and the CPU oracle: few and many survivors, one and several word segments per row,
samples, itemset limits, and searches without room in its arenas."""
import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import fim, synth

pytestmark = pytest.mark.gpu


def odict(o):
    so, si, sp = o
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


def groups(seed, D, sizes, share, noise):
    """Transactions that hold most items of one of several groups: frequent itemsets up to a group's size."""
    rng = np.random.default_rng(seed)
    start = np.concatenate([[0], np.cumsum(sizes)])
    N = int(start[-1])
    tx = []
    for _ in range(D):
        g = rng.integers(len(sizes))
        items = start[g] + np.nonzero(rng.random(sizes[g]) < share)[0]
        tx.append(np.unique(np.concatenate([items, rng.choice(N, size=min(N, rng.poisson(noise)), replace=False)])))
    off = np.concatenate([[0], np.cumsum([len(v) for v in tx])]).astype(np.uint32)
    return off, np.concatenate(tx).astype(np.uint32), N


CASES = {
    "three_rows": (lambda: groups(1, 300, [3], 0.8, 0.0), 60),
    "most_rows": (lambda: groups(2, 4_000, [3] * 341, 0.9, 1.0), 3),      # 1,023 rows, two or three survivors
    "few_survivors": (lambda: groups(3, 3_000, [6] * 40, 0.85, 1.0), 25),   # up to five: counted with their node
    "many_survivors": (lambda: groups(4, 2_000, [40] * 2, 0.4, 0.5), 50),  # more than eight candidates a node
    "wide_rows": (lambda: groups(5, 70_000, [9] * 4, 0.7, 0.5), 4_000),     # several segments of 512 words
    "deep": (lambda: groups(6, 1_200, [13] * 2, 0.97, 0.2), 250),
}


@pytest.mark.parametrize("name", CASES)
def test_same_search_as_frame_passes(name):
    make, minsup = CASES[name]
    off, items, N = make()
    want = odict(oracle.eclat(off, items, N, minsup))
    db = fim.build_vertical_db(off, items, N)
    try:
        got = db.mine(minsup, class_work=True)
        ref = db.mine(minsup, dfs_mode=fim.FIM_DFS_FRAMES, class_work=True)
        assert got.as_dict() == want and ref.as_dict() == want
        assert (got.stats["search"], got.stats["search_runs"]) == (fim.FIM_SEARCH_LEVELS, 1)
        assert ref.stats["search"] == fim.FIM_DFS_FRAMES
        for key in ("n_intersections", "n_classes", "n_queue_entries", "n_frequent", "n_items_out", "max_len", "bytes_dfs_kernel"):
            assert got.stats[key] == ref.stats[key], key
        assert np.array_equal(got.class_work, ref.class_work)
        assert any(len(k) >= 3 for k in want)
    finally:
        db.free()


@pytest.mark.parametrize("room", [dict(queue=1), dict(queue=20), dict(words=1), dict(words=100)], ids=str)
@pytest.mark.parametrize("name", ["many_survivors", "wide_rows", "deep"])
def test_without_room(name, room):
    """A search that finds no room in its arenas is repeated by the frame passes."""
    make, minsup = CASES[name]
    off, items, N = make()
    want = odict(oracle.eclat(off, items, N, minsup))
    db = fim.build_vertical_db(off, items, N)
    try:
        got = db.mine(minsup, class_work=True)
        got2 = db.mine(minsup, class_work=True, walk=room)
        assert (got.stats["search"], got.stats["search_runs"]) == (fim.FIM_SEARCH_LEVELS, 1)
        assert (got2.stats["search"], got2.stats["search_runs"]) == (fim.FIM_DFS_FRAMES, 2)
        assert got.as_dict() == want and got2.as_dict() == want
        for key in ("n_intersections", "n_classes", "n_queue_entries", "n_frequent", "n_items_out", "max_len"):
            assert got.stats[key] == got2.stats[key], key
        assert np.array_equal(got.class_work, got2.class_work)
    finally:
        db.free()


@pytest.mark.parametrize("words", [384, 416, 512, 544, 800, 832, 1_024, 1_056, 2_048, 2_080, 4_096, 4_128])
def test_row_lengths(words):
    """Rows at the edges of one, two, four and eight warps a unit and one or two segments, and of the one-pass subtrees."""
    off, items, N = groups(words, words * 32, [12, 4], 0.55, 0.2)
    minsup = words * 32 // 25
    db = fim.build_vertical_db(off, items, N)
    try:
        got = db.mine(minsup)
        ref = db.mine(minsup, dfs_mode=fim.FIM_DFS_FRAMES)
        assert got.as_dict() == ref.as_dict() == odict(oracle.eclat(off, items, N, minsup))
        assert got.stats["n_intersections"] == ref.stats["n_intersections"] and got.stats["max_len"] >= 4
        assert (got.stats["search"], got.stats["search_runs"]) == (fim.FIM_SEARCH_LEVELS, 1)
    finally:
        db.free()


@pytest.mark.parametrize("cost", ["itemsets", "intersections"])
@pytest.mark.parametrize("name", ["few_survivors", "many_survivors"])
def test_class_costs_of_a_sample(name, cost):
    make, minsup = CASES[name]
    off, items, N = make()
    D = len(off) - 1
    db = fim.build_vertical_db(off, items, N)
    try:
        want = oracle.class_costs(off, items, N, 0, 0.5, minsup / D, 9, kind=["itemsets", "intersections"].index(cost))
        got = db.estimate_class_costs(0.5, minsup / D, 9, cost=cost)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        db.estimate_class_costs(0.5, minsup / D, 9, cost=cost, outputs=False)
        got = db.estimate_result()
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    finally:
        db.free()


def test_many_itemsets_and_limits():
    """20 items in every one of 64 transactions: 2^20 - 1 itemsets in levels of up to 2^17.5; limits below and at the number
    of itemsets."""
    k, D = 20, 64
    off = (np.arange(D + 1) * k).astype(np.uint32)
    items = np.tile(np.arange(k, dtype=np.uint32), D)
    db = fim.build_vertical_db(off, items, k)
    try:
        r = db.mine(D, result_on_device=True)
        assert r.n_sets == 2 ** k - 1 and r.stats["max_len"] == k and r.stats["n_items_out"] == k * 2 ** (k - 1)
        assert r.stats["search"] == fim.FIM_SEARCH_LEVELS
        r.free()
        with pytest.raises(fim.FimError) as e:
            db.mine(D, max_itemsets=5_000)
        assert e.value.status == fim.FIM_ERR_OUTPUT_OVERFLOW
        off9, items9 = (np.arange(D + 1) * 9).astype(np.uint32), np.tile(np.arange(9, dtype=np.uint32), D)
    finally:
        db.free()
    db = fim.build_vertical_db(off9, items9, 9)
    try:
        assert db.mine(D, max_itemsets=511).n_sets == 511
        with pytest.raises(fim.FimError):
            db.mine(D, max_itemsets=510)
    finally:
        db.free()


def test_outgrown_search_is_not_tried_again():
    """A search by levels that outgrew its arenas is repeated by the frame passes once; further mines of the database at that
    minsup, and samples at theirs, take the frame passes at once, and mines that fit the levels again."""
    off, items = synth.dense_bernoulli(3, 20_000, 100)
    db = fim.build_vertical_db(off, items, 100)

    def launches(call):
        c = fim.kernel_launches()
        r = call()
        return fim.kernel_launches() - c, r

    try:
        def ran(ms, **kw):
            r = db.mine(ms, result_on_device=True, **kw)
            return r.n_sets, r.stats["search"], r.stats["search_runs"]

        n, _, runs = ran(7_600, dfs_mode=fim.FIM_DFS_FRAMES)
        assert ran(7_600) == (n, fim.FIM_DFS_FRAMES, runs + 1)
        assert ran(7_600) == (n, fim.FIM_DFS_FRAMES, runs)
        assert ran(7_500)[1:] == (fim.FIM_DFS_FRAMES, runs)
        assert ran(9_000)[:2] == (ran(9_000, dfs_mode=fim.FIM_DFS_FRAMES)[0], fim.FIM_SEARCH_LEVELS)
        first, e1 = launches(lambda: db.estimate_class_costs(1.0, 0.38, 5, max_sample_itemsets=0))
        second, e2 = launches(lambda: db.estimate_class_costs(1.0, 0.38, 5, max_sample_itemsets=0))
        assert second < first
        db.estimate_class_costs(1.0, 0.37, 5, max_sample_itemsets=0, outputs=False)  # (deferred)
        third, e3 = launches(db.estimate_result)
        assert third == 0
        for a, b in zip(e1, e2):
            assert np.array_equal(a, b)
    finally:
        db.free()
    db = fim.build_vertical_db(off, items, 100)
    try:  # the first deferred sample of a database: completed once, by the frame passes
        db.estimate_class_costs(1.0, 0.38, 5, max_sample_itemsets=0, outputs=False)
        redo, e4 = launches(db.estimate_result)
        assert 0 < redo <= second
        for a, b in zip(e1, e4):
            assert np.array_equal(a, b)
    finally:
        db.free()


def test_deferred_estimate_of_many_itemsets():
    """A deferred sample of 2^20 - 1 itemsets: the mine that uses it finds room for its result at once (k items alike:
    class i has 2^(k - 1 - i) itemsets)."""
    k, D = 20, 64
    db = fim.build_vertical_db((np.arange(D + 1) * k).astype(np.uint32), np.tile(np.arange(k, dtype=np.uint32), D), k)
    try:
        db.estimate_class_costs(1.0, 1.0, 3, outputs=False)
        r = db.mine(D, result_on_device=True)
        assert r.n_sets == 2 ** k - 1 and r.stats["search_runs"] == 1
        r.free()
        cost, order = db.estimate_result()[:2]
        assert np.array_equal(order, np.arange(k))
        assert np.allclose(cost, 2.0 ** np.arange(k - 1, -1, -1) / (2 ** k - 1), rtol=1e-12)
    finally:
        db.free()
