"""A caller built with the structs as they were before the last fields (GPU): served as before, nothing written past its
own counters."""
import ctypes

import numpy as np
import pytest

from paper_2108_05038_gb300 import fim

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("old", [False, True])
def test_counters_of_an_older_caller(old):
    rng = np.random.default_rng(1)
    tx = [np.nonzero(rng.random(20) < 0.4)[0] for _ in range(500)]
    off = np.concatenate([[0], np.cumsum([len(v) for v in tx])]).astype(np.uint32)
    db = fim.build_vertical_db(off, np.concatenate(tx).astype(np.uint32), 20)
    lib = fim.load()
    try:
        want = db.mine(60)
        n = ctypes.sizeof(fim.MineStats)
        room = (ctypes.c_uint8 * (n + 64))(*([0xA5] * (n + 64)))
        opts = fim.MineOpts()
        lib.fim_mine_opts_init(ctypes.byref(opts))
        known = fim.MineStats.pair_rows_tx.offset if old else n
        if old:
            opts.struct_size = fim.MineOpts.walk_queue.offset
            opts.walk_queue = opts.walk_words = opts.fault_plan_room = 1  # (past what it has: not read)
        opts.stats = ctypes.cast(room, ctypes.POINTER(fim.MineStats))
        h = ctypes.c_void_p()
        assert lib.fim_mine(db.handle, 60, ctypes.byref(opts), ctypes.byref(h)) == fim.FIM_OK
        assert fim.Result(lib, h.value, None).as_dict() == want.as_dict()
        got = fim.MineStats.from_buffer_copy(bytes(room[:n]))
        assert got.n_frequent == want.n_sets and got.n_intersections == want.stats["n_intersections"]
        assert bytes(room[known:]) == b"\xa5" * (n + 64 - known)
        plan = ctypes.c_void_p()
        assert lib.fim_plan_create(db.handle, 60, ctypes.byref(opts), ctypes.byref(plan)) == fim.FIM_OK
        assert lib.fim_plan_launch(plan) == fim.FIM_OK
        assert lib.fim_plan_result(plan, ctypes.byref(opts), ctypes.byref(h)) == fim.FIM_OK
        assert fim.Result(lib, h.value, None).as_dict() == want.as_dict()
        assert bytes(room[known:]) == b"\xa5" * (n + 64 - known)
        lib.fim_plan_free(plan)
    finally:
        db.free()
