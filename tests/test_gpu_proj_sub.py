"""The small-subtree walk of the projected DFS (GPU), against the sparse node mode (the same nodes, intersections and
class work) and the CPU oracle: parts of few and of many rows, subtrees past one round, parts too large for a warp."""
import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu


def odict(o):
    so, si, sp = o
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


def groups(seed, D, sizes, share, noise, repeat=1, lone=0):
    """Transactions that hold most items of one of several groups: frequent itemsets up to a group's size.  ``lone`` more
    items occur in one transaction each."""
    rng = np.random.default_rng(seed)
    start = np.concatenate([[0], np.cumsum(sizes)])
    N = int(start[-1])
    tx = []
    for _ in range(D):
        g = rng.integers(len(sizes))
        items = start[g] + np.nonzero(rng.random(sizes[g]) < share)[0]
        extra = rng.choice(N, size=rng.poisson(noise), replace=False)
        tx += [np.unique(np.concatenate([items, extra]))] * repeat
    for k in range(lone):
        tx[k % len(tx)] = np.append(tx[k % len(tx)], N + k)
    off = np.concatenate([[0], np.cumsum([len(v) for v in tx])]).astype(np.uint32)
    return off, np.concatenate(tx).astype(np.uint32), N + lone


CASES = {
    # (groups, minsup): many parts of 2-5 rows; of 6-32; of more than 32; subtrees of thousands of sets, past a round
    "few_rows": (lambda: groups(1, 4_000, [4] * 300, 0.9, 1.0), 6),
    "some_rows": (lambda: groups(2, 6_000, [9] * 130, 0.8, 2.0), 12),
    "many_rows": (lambda: groups(3, 3_000, [45] * 3, 0.35, 0.5), 60),
    "deep": (lambda: groups(4, 1_500, [15] * 4, 0.97, 0.5, lone=40), 200),
    # wide regions: parts past a warp's shared memory that get rows of their own, and (dense) that do not
    "wide": (lambda: groups(5, 60_000, [14] * 6, 0.5, 1.0), 900),
    "wide_dense": (lambda: groups(6, 40_000, [12], 0.8, 0.0), 9_000),
    "repeated_transactions": (lambda: groups(7, 500, [10] * 20, 0.7, 0.5, repeat=7), 20),
}


@pytest.mark.parametrize("name", CASES)
def test_same_walk_as_sparse_nodes(name):
    make, minsup = CASES[name]
    off, items, N = make()
    db = fim.build_vertical_db(off, items, N)
    try:
        ref = db.mine(minsup, dfs_mode=fim.FIM_DFS_SPARSE, class_work=True, class_order="uniform")
        got = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, class_work=True, class_order="uniform")
        want = odict(oracle.eclat(off, items, N, minsup))
        assert got.as_dict() == want and ref.as_dict() == want
        assert (got.stats["search"], got.stats["search_runs"]) == (fim.FIM_SEARCH_SUBTREES, 1)
        assert ref.stats["search"] == fim.FIM_DFS_SPARSE
        for key in ("n_intersections", "n_classes", "n_queue_entries", "n_frequent", "n_items_out", "max_len"):
            assert got.stats[key] == ref.stats[key], key
        assert np.array_equal(got.class_work, ref.class_work)
        assert any(len(k) >= 3 for k in want)
        top = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, output="maximal").as_dict()
        # maximal: no frequent superset of one item more
        covered = {k[:i] + k[i + 1:] for k in want for i in range(len(k))}
        assert top == {k: v for k, v in want.items() if k not in covered}
    finally:
        db.free()


# what the walk does without room: parts, subtrees' rests and their rows go to the projected DFS, or the run is repeated
# without the walk; a cycle per subtree hands on everything that can be
ROOMS = {
    "one_entry": dict(queue=1, cycles=1),
    "forty_entries": dict(queue=40, cycles=2_000),
    "some_entries": dict(queue=700, cycles=1),
    "no_words": dict(words=1, cycles=1),
    "some_words": dict(words=6_000, cycles=1),
    "one_round": dict(rounds=1, cycles=1),
    "three_rounds": dict(rounds=3, cycles=1),
    "all_rounds": dict(cycles=1),
}


@pytest.fixture(scope="module")
def searched():
    """The cases' databases, their itemsets and the sparse node mode's counters, made once."""
    made = {}

    def get(name):
        if name not in made:
            make, minsup = CASES[name]
            off, items, N = make()
            db = fim.build_vertical_db(off, items, N)
            ref = db.mine(minsup, dfs_mode=fim.FIM_DFS_SPARSE, class_work=True, class_order="uniform")
            want = odict(oracle.eclat(off, items, N, minsup))
            assert ref.as_dict() == want
            made[name] = db, minsup, want, ref
        return made[name]

    yield get
    for db, *_ in made.values():
        db.free()


@pytest.mark.parametrize("room", ROOMS)
@pytest.mark.parametrize("name", ["many_rows", "deep", "wide", "wide_dense"])
def test_without_room(searched, name, room):
    db, minsup, want, ref = searched(name)
    got = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, class_work=True, class_order="uniform", walk=ROOMS[room])
    assert got.as_dict() == want
    assert (got.stats["search"], got.stats["search_runs"]) in ((fim.FIM_SEARCH_SUBTREES, 1), (fim.FIM_DFS_PROJECTED, 2))
    for key in ("n_intersections", "n_classes", "n_queue_entries", "n_frequent", "n_items_out", "max_len"):
        assert got.stats[key] == ref.stats[key], key
    assert np.array_equal(got.class_work, ref.class_work)
    top = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, output="maximal", walk=ROOMS[room]).as_dict()
    covered = {k[:i] + k[i + 1:] for k in want for i in range(len(k))}
    assert top == {k: v for k, v in want.items() if k not in covered}


def test_large_subtree_without_room():
    """27 items in every one of 64 transactions, queues of one entry: a part with 2^25 itemsets below it finds no room for
    its rest in the next round, and is shared by the warps of the projected DFS all the same."""
    k, D = 27, 64
    db = fim.build_vertical_db((np.arange(D + 1) * k).astype(np.uint32), np.tile(np.arange(k, dtype=np.uint32), D), k)
    try:
        for walk in (dict(), dict(queue=1)):
            r = db.mine(D, dfs_mode=fim.FIM_DFS_PROJECTED, result_on_device=True, walk=walk)
            assert r.n_sets == 2 ** k - 1 and r.stats["max_len"] == k and r.stats["n_items_out"] == k * 2 ** (k - 1)
            r.free()
    finally:
        db.free()


@pytest.mark.parametrize("words", [3_000, 20_000, 100_000])
@pytest.mark.parametrize("name", ["many_rows", "deep"])
def test_hand_out_without_room(searched, name, words):
    """Frames that the projected DFS would hand to other warps (all of three survivors or more) where the arena has no room
    for their database parts: the warps keep them, and the slots reserved for them are passed over."""
    db, minsup, want, ref = searched(name)
    got = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, class_work=True, class_order="uniform", proj_split_words=1,
                  proj_bitmap_words=words, walk=dict(words=1))
    assert got.as_dict() == want and got.stats["search"] == fim.FIM_DFS_PROJECTED and got.stats["n_proj_classes"] > 0
    for key in ("n_intersections", "n_classes", "n_queue_entries", "n_frequent", "n_items_out", "max_len"):
        assert got.stats[key] == ref.stats[key], key
    assert np.array_equal(got.class_work, ref.class_work)


def test_class_bitmaps_past_32_bit_offsets(searched):
    """With a budget that lets a class region hold 2^32 words the walk, whose row offsets have 32 bits, is left out."""
    db, minsup, want, ref = searched("many_rows")
    for words, search in ((1 << 24, fim.FIM_SEARCH_SUBTREES), ((1 << 32) - 1, fim.FIM_SEARCH_SUBTREES),
                          (1 << 32, fim.FIM_DFS_PROJECTED)):
        got = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED, proj_bitmap_words=words, walk=dict(words=100_000))
        assert got.as_dict() == want and got.stats["n_intersections"] == ref.stats["n_intersections"]
        assert (got.stats["search"], got.stats["search_runs"]) == (search, 1)


@pytest.mark.parametrize("limit", [50, 2_000])
def test_itemset_limit_stops_the_walk(limit):
    off, items, N = CASES["deep"][0]()
    db = fim.build_vertical_db(off, items, N)
    try:
        with pytest.raises(fim.FimError) as e:
            db.mine(200, dfs_mode=fim.FIM_DFS_PROJECTED, max_itemsets=limit)
        assert e.value.status == fim.FIM_ERR_OUTPUT_OVERFLOW
        n = db.mine(200, dfs_mode=fim.FIM_DFS_PROJECTED).n_sets
        assert n == db.mine(200, dfs_mode=fim.FIM_DFS_PROJECTED, max_itemsets=n).n_sets
    finally:
        db.free()


def test_plan_replays_the_walk():
    """The walk's launch inside a captured graph."""
    off, items, N = CASES["some_rows"][0]()
    db = fim.build_vertical_db(off, items, N)
    try:
        want = db.mine(12, dfs_mode=fim.FIM_DFS_PROJECTED).as_dict()
        plan = db.plan(12, dfs_mode=fim.FIM_DFS_PROJECTED)
        for _ in range(3):
            plan.launch()
            assert plan.result().as_dict() == want
        plan.free()
    finally:
        db.free()
