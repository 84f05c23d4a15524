"""fim_extension_supports over its launch shapes (GPU): few to many candidates (8, 4, 2 or 1 warps per candidate, and more
candidates than can be resident), prefixes ANDed inside the counting kernel and before it, repeated candidates."""
import numpy as np
import pytest

from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu

N, D = 9_500, 2_100


@pytest.fixture(scope="module")
def case():
    rng = np.random.default_rng(8)
    m = rng.random((D, N)) < 0.01
    m[:, :300] = rng.random((D, 300)) < 0.9  # items that prefixes of several hundred still share
    off = np.concatenate([[0], np.cumsum(m.sum(1))]).astype(np.uint32)
    db = fim.build_vertical_db(off, np.nonzero(m)[1].astype(np.uint32), N)
    yield m, db
    db.free()


@pytest.mark.parametrize("n_prefix", [1, 2, 8, 9, 260])
@pytest.mark.parametrize("n_cand", [1, 7, 912, 1_300, 1_825, 3_649, 7_296, 7_297, 9_500])
def test_counts(case, n_cand, n_prefix):
    m, db = case
    rng = np.random.default_rng(n_cand + n_prefix)
    prefix = rng.choice(300, n_prefix, replace=False)
    cand = rng.integers(0, N, n_cand)
    want = m[m[:, prefix].all(1)].sum(0)[cand]
    assert np.array_equal(db.extension_supports(prefix, cand), want)


def test_large_rows_take_the_prefix_kernel():
    """A prefix whose rows are too many bytes to be read again for every candidate."""
    rng = np.random.default_rng(3)
    D, N = 400_000, 700
    m = rng.integers(0, N, (D, 4))
    m[:, 0] = rng.integers(0, 3, D)
    m = np.sort(m, axis=1)
    off = (np.arange(D + 1) * 4).astype(np.uint32)
    db = fim.build_vertical_db(off, m.reshape(-1).astype(np.uint32), N)
    has = (m == 0).any(1) & (m == 5).any(1) & (m == 6).any(1)
    two = (m == 0).any(1) & (m == 5).any(1)
    for prefix, rows in (([0, 5], two), ([0, 5, 6], has)):
        want = np.array([(m[rows] == c).any(1).sum() for c in range(N)])
        assert np.array_equal(db.extension_supports(prefix, np.arange(N)), want)
    db.free()
