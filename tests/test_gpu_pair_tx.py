"""Level 2 counted from the transactions (GPU): the automatic choice on sparse data, for all rows or for all but the
256 most frequent, against the integer-pipe kernel on the same database and the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu


def database(seed, D, N, lengths, hot=0):
    """Transactions of the given lengths (cycled) of distinct items; each of the last ``hot`` items is also put into
    half of the transactions (so that their pairs are the many)."""
    rng = np.random.default_rng(seed)
    tx = []
    for t in range(D):
        n = lengths[t % len(lengths)]
        items = rng.choice(N - hot, size=n, replace=False)
        if hot:
            items = np.concatenate([items, N - hot + np.nonzero(rng.random(hot) < 0.5)[0]])
        tx.append(rng.permutation(items))
    off = np.concatenate([[0], np.cumsum([len(v) for v in tx])]).astype(np.uint32)
    return off, np.concatenate(tx).astype(np.uint32)


def odict(o):
    so, si, sp = o
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


def check(off, items, N, minsup, kernel, left=0, want=None, **kw):
    """``left``: rows whose pairs another kernel (``kernel``) counts from the rows."""
    db = fim.build_vertical_db(off, items, N, **kw)
    try:
        auto = db.mine(minsup)
        assert auto.stats["pair_kernel"] == kernel
        assert auto.stats["pair_rows_tx"] == auto.stats["n_frequent_items"] - left
        cores = db.mine(minsup, pair_kernel=fim.FIM_PAIR_CORES)
        assert cores.stats["pair_kernel"] == fim.FIM_PAIR_CORES and cores.stats["pair_rows_tx"] == 0
        got = auto.as_dict()
        assert got == cores.as_dict()
        if want is not None:
            assert got == want
        return got
    finally:
        db.free()


@pytest.mark.parametrize("D", [4001, 20_000, 77_777])
@pytest.mark.parametrize("N,lengths", [
    (1200, [0, 1, 2, 3, 4, 5]),               # empty and single-item transactions, odd and even pairings
    (1500, [2] * 30 + [31, 32, 33]),          # the edges of one 32-item chunk
    (3001, [1] * 60 + [64, 65, 96, 100]),     # long transactions: pairs across chunks
])
def test_pairs_from_transactions(D, N, lengths):
    off, items = database(D + N, D, N, lengths)
    k = np.diff(off.astype(np.int64))
    mean = float((k * (k - 1)).sum()) / (N * (N - 1))  # of a pair's support: the minsup is some deviations above it
    minsup = max(2, int(mean + 2.5 * mean ** 0.5) + 1)
    got = check(off, items, N, minsup, fim.FIM_PAIR_CORES, 0,
                odict(oracle.eclat(off, items, N, minsup)) if D < 10_000 else None)
    assert any(len(k) == 2 for k in got)


@pytest.mark.parametrize("N", [1100, 1280, 1281, 2047])
def test_most_frequent_rows_left_to_the_product(N):
    """Rows that all take part, with the last ones so frequent that the product counts their pairs."""
    off, items = database(N, 100_000, N, [3, 4, 5], hot=8)
    minsup = 100
    got = check(off, items, N, minsup, fim.FIM_PAIR_TENSOR_FUSED, 256)
    assert any(len(k) == 2 for k in got)


def test_repeated_items_take_the_rows():
    """A transaction that holds an item twice counts it once, in supports and in pairs."""
    off, items = database(5, 20_000, 1200, [4])
    items = items.copy()
    items[3::4] = items[2::4]  # the last item of every transaction repeats the one before it
    want = odict(oracle.eclat(off, items, 1200, 20))
    db = fim.build_vertical_db(off, items, 1200)
    try:
        got = db.mine(20)
        assert got.as_dict() == want and got.stats["pair_rows_tx"] == 0
    finally:
        db.free()


@pytest.mark.parametrize("prefilter", [0, 8])
def test_noalloc_pairs_from_transactions(prefilter):
    """(That call reports no counters.  It chooses between the transactions and the integer pipes by the model of a mine's
    choice, which has the tensor cores as well, and a mine of the same rows takes the transactions here.)"""
    import torch

    off, items = database(11, 60_000, 1000, [1] * 20 + [3, 8, 33])
    db = fim.build_vertical_db(off, items, 1000, prefilter_minsup=prefilter)
    try:
        assert db.mine(8).stats["pair_rows_tx"] == 1000
        want = {k: v for k, v in db.mine(8, pair_kernel=fim.FIM_PAIR_CORES).as_dict().items() if len(k) == 2}
        p = torch.zeros(len(want) + 1, 2, dtype=torch.int32, device="cuda")
        s = torch.zeros(len(want) + 1, dtype=torch.int32, device="cuda")
        n = db.mine_pairs_noalloc(8, p, s, len(want) + 1)
        got = {tuple(k): v for k, v in zip(p[:n].tolist(), s[:n].tolist())}
        assert got == want
    finally:
        db.free()


@pytest.mark.parametrize("N,D", [(5000, 40_000), (1200, 40_000)])
def test_sample_pairs_from_transactions(N, D):
    """The estimate's sample, over a choice of the rows (N = 5000) or over all of them, drawn with replacement (whichever
    kernel the model takes for it: an estimate reports no counters)."""
    off, items = database(N, D, N, [2, 5, 9, 33])
    rel = 12 / D
    db = fim.build_vertical_db(off, items, N)
    try:
        for rate in (0.02, 0.25):
            cost, order = db.estimate_class_costs(rate, rel, 3)
            ocost, oorder, _ = oracle.class_costs(off, items, N, 0, rate, rel, 3)
            assert np.array_equal(cost, ocost) and np.array_equal(order, oorder)
    finally:
        db.free()
