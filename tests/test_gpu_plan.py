"""Batched plans (one persistent launch captured in a CUDA graph) and the
launch-shape autotuner, against the CPU oracle: bit-exact, replay after replay."""
import numpy as np
import pytest

import oracle
from paper_2108_05038_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2108_05038_gb300 import fim  # noqa: E402


def odict(res):
    so, si, sp = res
    return {tuple(int(v) for v in si[so[k]:so[k + 1]]): int(sp[k]) for k in range(len(sp))}


@pytest.mark.parametrize("name,D", [("dense_deep", 50_000), ("tiny", 10_000), ("sparse_mid", 40_000)])
def test_plan_replays_match_oracle(name, D):
    w = synth.make_workload(name, D=D)
    ms = synth.abs_minsup(w["rel_minsup"], D)
    want = odict(oracle.eclat(w["offsets"], w["items"], w["N"], ms))
    db = fim.build_vertical_db(w["offsets"], w["items"], w["N"])
    db.estimate_class_costs(0.02 if D >= 40_000 else 0.1, w["rel_minsup"], 11)
    plan = db.plan(ms)
    for _ in range(3):
        plan.launch()
        res = plan.result()
        assert res.as_dict() == want
    for _ in range(4):  # back-to-back replays, one result at the end
        plan.launch()
    assert plan.result().as_dict() == want
    plan.free()
    db.free()


def test_plan_on_torch_stream_and_device_result():
    w = synth.make_workload("dense_deep", D=20_000)
    ms = 12_000
    want = odict(oracle.eclat(w["offsets"], w["items"], w["N"], ms))
    s = torch.cuda.Stream()
    db = fim.build_vertical_db(w["offsets"], w["items"], w["N"], stream=s)
    plan = db.plan(ms, result_on_device=True)
    assert plan.stream == s.cuda_stream
    plan.launch()
    res = plan.result(result_on_device=True)
    assert res.on_device and res.n_sets == len(want)
    plan.free()
    db.free()


def test_autotune_shape_is_valid_and_output_unchanged():
    w = synth.make_workload("dense_deep", D=30_000)
    ms = 18_000
    want = odict(oracle.eclat(w["offsets"], w["items"], w["N"], ms))
    db = fim.build_vertical_db(w["offsets"], w["items"], w["N"])
    shape, best_ms = db.autotune(ms)
    assert shape["threads_per_cta"] in (128, 256, 512) and shape["vec_per_lane"] in (1, 2, 4, 8)
    assert best_ms > 0
    again, ms2 = db.autotune(ms)  # cached
    assert again == shape and ms2 == best_ms
    assert db.mine(ms, shape=shape).as_dict() == want
    plan = db.plan(ms, shape=shape)
    plan.launch()
    assert plan.result().as_dict() == want
    plan.free()
    db.free()


def test_autotune_times_the_automatic_traversal_too():
    """On a dense database of few rows the search by levels, which only the automatic choice takes, is the fastest."""
    w = synth.make_workload("dense_deep", D=50_000)
    ms = synth.abs_minsup(w["rel_minsup"], 50_000)
    db = fim.build_vertical_db(w["offsets"], w["items"], w["N"])
    try:
        shape, best_ms = db.autotune(ms)
        auto = min(db.mine(ms, collect_times=True).stats["ms_device_total"] for _ in range(5))
        frames = min(db.mine(ms, collect_times=True, dfs_mode=fim.FIM_DFS_FRAMES).stats["ms_device_total"] for _ in range(5))
        assert auto < frames
        assert shape["dfs_mode"] == fim.FIM_DFS_AUTO and best_ms < frames
    finally:
        db.free()


@pytest.mark.parametrize("mode", [None, fim.FIM_DFS_PROJECTED])
def test_replay_without_room_is_repeated(mode):
    """Replays whose search by levels, or small-subtree walk, has no room (the sizing run has it): the first result comes
    from a repeated run, and the plan is captured anew for the launches after it."""
    rng = np.random.default_rng(8)
    D, k = 3_000, 45
    tx = [np.nonzero(rng.random(k) < 0.35)[0] for _ in range(D)]
    off = np.concatenate([[0], np.cumsum([len(v) for v in tx])]).astype(np.uint32)
    items = np.concatenate(tx).astype(np.uint32)
    want = odict(oracle.eclat(off, items, k, 60))
    db = fim.build_vertical_db(off, items, k)
    kw = {} if mode is None else {"dfs_mode": mode}
    try:
        plan = db.plan(60, fault_plan_room=True, **kw)
        counts = []
        for _ in range(3):
            c = fim.kernel_launches()
            plan.launch()
            plan.launch()
            res = plan.result()
            assert res.as_dict() == want
            counts.append((fim.kernel_launches() - c, res.stats["search_runs"], res.stats["search"]))
        without = fim.FIM_DFS_FRAMES if mode is None else fim.FIM_DFS_PROJECTED
        assert counts[0][0] > counts[1][0] and counts[1] == counts[2] == (counts[1][0], 1, without)
        assert counts[0][1:] == (2, without)
        plan.free()
        assert db.mine(60, **kw).as_dict() == want
    finally:
        db.free()


def test_launch_counter_counts_graph_kernels_per_replay():
    """fim_kernel_launches: a mine adds its kernels; each plan replay adds the kernels of its graph."""
    w = synth.make_workload("dense_deep", D=20_000)
    ms = 12_000
    db = fim.build_vertical_db(w["offsets"], w["items"], w["N"])
    c0 = fim.kernel_launches()
    db.mine(ms).free()
    c1 = fim.kernel_launches()
    assert c1 - c0 >= 5  # pair counts, survivor count, level-2 scan and fill, DFS
    plan = db.plan(ms)
    c2 = fim.kernel_launches()
    plan.launch()
    c3 = fim.kernel_launches()
    plan.launch()
    plan.launch()
    c4 = fim.kernel_launches()
    assert c3 - c2 >= 5 and c4 - c3 == 2 * (c3 - c2)
    plan.result().free()
    plan.free()
    db.free()
