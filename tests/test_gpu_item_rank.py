"""The build's row order (GPU): items ranked on the device (up to 16,384 of them) or sorted on the host, with and without a
prefilter, against a stable sort of the counts; a database that the item count finds invalid is refused and the next one built."""
import numpy as np
import pytest

from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu


def database(seed, N, D):
    rng = np.random.default_rng(seed)
    length = rng.integers(0, min(N, 6) + 1, D)
    tx = [np.sort(rng.choice(N, size=n, replace=False)) for n in length]
    off = np.concatenate([[0], np.cumsum(length)]).astype(np.uint32)
    return off, (np.concatenate(tx) if off[-1] else np.zeros(0)).astype(np.uint32)


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("prefilter", [0, 1, 2])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 33, 1000, 16_384, 16_385])
def test_rows_by_support_then_id(N, prefilter, device):
    D = 3_000
    off, items = database(N, N, D)
    if device:
        import torch
        d = [torch.from_numpy(a.view(np.int32)).cuda() for a in (off, items)]
        db = fim.build_vertical_db_device(*d, D, N, prefilter_minsup=prefilter)
    else:
        db = fim.build_vertical_db(off, items, N, prefilter_minsup=prefilter)
    cnt = np.bincount(items, minlength=N)
    order = np.argsort(cnt, kind="stable")
    order = order[cnt[order] >= prefilter]
    rows, supp = db.rows()
    assert np.array_equal(rows, order) and np.array_equal(supp, cnt[order])
    top = int(order[-1])
    assert db.extension_supports([top], [top])[0] == cnt[top]
    db.free()


def test_invalid_input_leaves_the_next_build_sound():
    off, items = database(3, 50, 500)
    bad = items.copy()
    bad[7] = 50
    with pytest.raises(fim.FimError):
        fim.build_vertical_db(off, bad, 50)
    import torch
    torch.cuda.synchronize()
    db = fim.build_vertical_db(off, items, 50)
    cnt = np.bincount(items, minlength=50)
    assert np.array_equal(db.extension_supports([int(np.argmax(cnt))], [int(np.argmax(cnt))]), [cnt.max()])
    db.free()
