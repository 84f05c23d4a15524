"""The transactions of a class in projected mode (GPU): rows of few, many and nearly all bits, at the edges of the rounds that
list them (256 words a warp, four to sixteen warps a row), against the CPU oracle."""
import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu


def odict(o):
    so, si, sp = o
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


@pytest.mark.parametrize("words", [1, 256, 257, 1_024, 1_056, 4_096, 4_128])
def test_rows_of_every_density(words):
    D = 32 * words - 5
    rng = np.random.default_rng(words)
    share = np.array([0.004, 0.02, 0.2, 0.25, 0.3, 0.6, 0.95, 1.0])
    M = rng.random((D, share.size)) < share
    M[:, 0] |= rng.random(D) < 0.01 * M[:, 1]
    off = np.concatenate([[0], np.cumsum(M.sum(1))]).astype(np.uint32)
    items = np.nonzero(M)[1].astype(np.uint32)
    minsup = max(2, D // 300)
    db = fim.build_vertical_db(off, items, share.size)
    try:
        got = db.mine(minsup, dfs_mode=fim.FIM_DFS_PROJECTED)
        assert got.as_dict() == odict(oracle.eclat(off, items, share.size, minsup))
        assert got.stats["n_proj_classes"] > 0
    finally:
        db.free()
