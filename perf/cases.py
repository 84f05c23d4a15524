"""The work that a user of this framework has it do, as cases to time.

A case is a dict of plain values.  ``kind`` is the call a program makes:

* ``step``    a database arrives as CSR (host arrays or device tensors), its class costs are estimated from the
              1% sample and it is mined once: build + estimate + mine, the framework's main path;
* ``mine``    another mine of a database that stays resident (a new output kind or minsup for the same data);
* ``plan``    the replay of a mine captured in a CUDA graph, with its result;
* ``extend``  the supports of P u {c} for a list of candidates c (a query against a resident database);
* ``pairs``   the frequent pairs into caller-owned buffers, without an allocation;
* ``serve``   a burst of mining jobs through the continuous-batching server.

Databases follow the laws of ``synth`` (pattern-embedded with uniform or Zipf item popularity, or dense Bernoulli).
Records of a result have no set order, so they are put in one when they are read for a comparison (``Read``): a
program that uses them would not sort them, and the pass ends with the result in its hands.  There they are also
padded to a length that the law sets, since how many there are depends on the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_05038_gb300 import fim, synth

SAMPLE_RATE = 0.01   # the 1% sample of the class-cost estimate
JOB_LIMIT = 4_000_000  # itemsets of a served job, past which it is refused


def listed():
    return [
        # the smallest whole call: ten thousand transactions from host memory, where launches and waits are all
        dict(name="step_tiny", kind="step", law="uniform", D=10_000, N=100, TL=10.0, PL=4.0, rel=0.01, word_bits=32,
             host=True, costs=False, prefilter=False),
        # an ordinary sparse database already on the device
        dict(name="step_sparse_mid", kind="step", law="uniform", D=100_000, N=1_000, TL=10.0, PL=4.0, rel=0.0025,
             word_bits=64, host=False, costs=False, prefilter=False),
        # dense data with long transactions: few items, a deep search
        dict(name="step_dense", kind="step", law="dense", D=50_000, N=75, TL=46.9, PL=0.0, rel=0.6, word_bits=64,
             host=False, costs=False, prefilter=False),
        # the benchmark's workload: a million transactions, Zipf items, 1.4 million itemsets
        dict(name="step_large", kind="step", law="zipf", D=1_000_000, N=10_000, TL=20.0, PL=6.0, rel=0.0005,
             word_bits=64, host=False, costs=False, prefilter=False),
        # odd sizes from host memory, infrequent items dropped at the build, the class costs read by the program
        dict(name="step_ragged", kind="step", law="uniform", D=299_993, N=3_331, TL=13.0, PL=4.0, rel=0.003,
             word_bits=32, host=True, costs=True, prefilter=True),
        # the maximal itemsets of a resident database of the benchmark's laws
        dict(name="mine_maximal", kind="mine", law="zipf", D=70_001, N=10_000, TL=20.0, PL=6.0, rel=0.001,
             word_bits=64, output="maximal", on_device=False),
        # the closed itemsets of a wider one, left on the device
        dict(name="mine_closed", kind="mine", law="zipf", D=200_000, N=10_000, TL=20.0, PL=6.0, rel=0.0005,
             word_bits=64, output="closed", on_device=True),
        # the batched form: one captured mine replayed, as when the same classes are mined again and again
        dict(name="plan_dense", kind="plan", law="dense", D=50_000, N=75, TL=46.9, PL=0.0, rel=0.6, word_bits=64),
        # a query with a short answer: the latency of one call
        dict(name="extend_small", kind="extend", law="strata", D=100_000, N=1_000, TL=10.0, prefix=2, candidates=1_000),
        # a query that streams every row of a large database
        dict(name="extend_large", kind="extend", law="strata", D=1_000_000, N=4_001, TL=20.0, prefix=1,
             candidates=4_001),
        # the frequent pairs of a database of as many items as that entry point takes
        dict(name="pairs_mid", kind="pairs", law="uniform", D=100_000, N=1_000, TL=10.0, PL=4.0, rel=0.0025,
             word_bits=64),
        # twelve jobs of the serving law that arrive together, four slots
        dict(name="serve_burst", kind="serve", jobs=12, D_lo=10_000, D_hi=200_000, N_lo=100, N_hi=5_000, rel_lo=0.005,
             rel_hi=0.05, slots=4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _pattern(rng, law, D_lo, D_hi):
    """A sparse database's law.  Minsups keep the frequent itemsets near those of the listed cases: pairs of
    independent items (share (TL / N)^2) stay rare, which is what a sparse database's user asks for."""
    D = int(_log(rng, D_lo, D_hi))
    if law == "uniform":
        N = int(_log(rng, 100, 5_000))
        TL = round(rng.uniform(5.0, 16.0), 1)
        rel = max(round(_log(rng, 0.0025, 0.02), 5), round(1.0 * (TL / N) ** 2, 5), round(60.0 / D, 5))
        PL = 4.0
    else:
        N = int(_log(rng, 4_000, 10_000))
        TL = round(rng.uniform(8.0, 18.0), 1)
        rel = max(round(_log(rng, 0.001, 0.01), 5), round(60.0 / D, 5))
        PL = 6.0
    return dict(law=law, D=D, N=N, TL=TL, PL=PL, rel=rel, word_bits=rng.choice([32, 64]))


def _dense(rng):
    D = int(_log(rng, 5_000, 100_000))
    return dict(law="dense", D=D, N=rng.randint(40, 90), TL=46.9, PL=0.0, rel=round(rng.uniform(0.58, 0.75), 3),
                word_bits=rng.choice([32, 64]))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "mine", "mine", "plan", "extend", "extend", "pairs", "serve"])
    if kind == "step":
        law = rng.choice(["uniform", "uniform", "zipf", "dense"])
        c = _dense(rng) if law == "dense" else _pattern(rng, law, 10_000 if law == "uniform" else 50_000, 900_000)
        return dict(kind=kind, **c, host=rng.random() < 0.5, costs=rng.random() < 0.3, prefilter=rng.random() < 0.3)
    if kind == "mine":
        c = _pattern(rng, rng.choice(["uniform", "zipf"]), 20_000, 300_000)
        return dict(kind=kind, **c, output=rng.choice(["all", "maximal", "closed"]), on_device=rng.random() < 0.5)
    if kind == "plan":
        return dict(kind=kind, **(_dense(rng) if rng.random() < 0.5 else _pattern(rng, "uniform", 10_000, 100_000)))
    if kind == "extend":
        N = int(_log(rng, 100, 4_000))
        return dict(kind=kind, law="strata", D=int(_log(rng, 10_000, 1_000_000)), N=N,
                    TL=float(rng.randint(5, min(20, N // 5))), prefix=rng.randint(1, 3), candidates=rng.randint(N // 8, N))
    if kind == "pairs":
        c = _pattern(rng, "uniform", 10_000, 300_000)
        return dict(kind=kind, **dict(c, N=min(c["N"], rng.randint(100, 1_000))))
    D_lo = int(_log(rng, 10_000, 50_000))
    return dict(kind="serve", jobs=rng.randint(2, 12), D_lo=D_lo, D_hi=4 * D_lo, N_lo=100, N_hi=rng.randint(500, 5_000),
                rel_lo=0.005, rel_hi=0.05, slots=rng.choice([1, 2, 4]))


# ---------------------------------------------------------------------------
# inputs


def _database(case, seed):
    """Host CSR (uint32 offsets, items) of the case's law."""
    if case["law"] == "dense":
        return synth.dense_bernoulli(seed, case["D"], case["N"])
    return synth.pattern_db(seed, case["D"], case["N"], case["TL"], case["PL"], 2 * case["N"],
                            "zipf" if case["law"] == "zipf" else "uniform")


def _strata(case, seed):
    """Device CSR (int32) with one item of each of TL equal strata of the items per transaction: distinct
    ascending ids, the first stratum's ids (a query's prefix is taken there) far more frequent than the others."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    D, N, TL = case["D"], case["N"], int(case["TL"])
    edge = torch.arange(TL + 1, device="cuda", dtype=torch.int64) * N // TL
    u = torch.rand(D, TL, generator=g, device="cuda")
    u[:, 0] = u[:, 0] ** 8
    items = (edge[:-1] + (u * (edge[1:] - edge[:-1])).long().clamp_(max=edge[1] - 1)).to(torch.int32)
    off = (torch.arange(D + 1, device="cuda", dtype=torch.int64) * TL).to(torch.int32)
    return off, items.reshape(-1).contiguous()


def _minsup(case):
    return synth.abs_minsup(case["rel"], case["D"])


def _on_device(a):
    return torch.from_numpy(a.view(np.int32)).cuda()


def _jobs(case, seed):
    st = seed * 7919 + 17

    def unit(k):
        return (synth.splitmix64_stream((st + k) & (2 ** 64 - 1), 1)[0] >> 11) / 9007199254740992.0

    jobs = []
    for k in range(case["jobs"]):
        # sizes and minsups spread evenly over their ranges, in an order that is not that of size
        x, y = (k * 5 % case["jobs"] + 0.5) / case["jobs"], (k * 7 % 12 + 0.5) / 12.0
        D = int(case["D_lo"] * (case["D_hi"] / case["D_lo"]) ** x)
        N = int(case["N_lo"] + (case["N_hi"] - case["N_lo"]) * unit(4 * k))
        TL = min(5.0 + 25.0 * unit(4 * k + 1), N / 10.0)
        rel = case["rel_lo"] * (case["rel_hi"] / case["rel_lo"]) ** y
        off, items = synth.pattern_db((seed + k) * 131 + 5, D, N, TL, 4.0, 2 * N, "uniform")
        jobs.append((off, items, N, max(1, math.ceil(max(rel, 0.8 * (TL / N) ** 2) * D))))
    return jobs


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "serve":
        s["jobs"] = _jobs(case, seed)
        s["server"] = fim.Server(0, case["slots"], 1, JOB_LIMIT)
        return s
    if kind == "extend":
        off, items = _strata(case, seed)
        s["db"] = fim.build_vertical_db_device(off, items, case["D"], case["N"])
        rng = np.random.RandomState(seed % (1 << 31))
        # a prefix that occurs: items of one transaction, the most frequent one first
        row = items[: int(case["TL"])].cpu().numpy().astype(np.uint32)
        s["prefix"] = np.concatenate([np.zeros(1, np.uint32), row[1:case["prefix"]]])
        s["candidates"] = np.sort(rng.permutation(case["N"])[: case["candidates"]]).astype(np.uint32)
        torch.cuda.synchronize()
        return s
    off, items = _database(case, seed)
    s["minsup"] = _minsup(case)
    if kind == "step":
        if case["host"]:
            s["off"], s["items"] = off, items
        else:
            s["off"], s["items"] = _on_device(off), _on_device(items)
        return s
    s["db"] = fim.build_vertical_db(off, items, case["N"], word_bits=case["word_bits"])
    if kind == "pairs":
        n = case["N"] * (case["N"] - 1) // 2
        s["pairs"] = torch.zeros(n, 2, dtype=torch.int32, device="cuda")
        s["supports"] = torch.zeros(n, dtype=torch.int32, device="cuda")
        return s
    s["db"].estimate_class_costs(SAMPLE_RATE, case["rel"], seed=1)
    if kind == "plan":
        s["plan"] = s["db"].plan(s["minsup"])
    return s


# ---------------------------------------------------------------------------
# one pass


class _DeviceArray:
    """A device result's array, for torch.as_tensor."""

    def __init__(self, ptr, n, typestr):
        self.__cuda_array_interface__ = dict(shape=(n,), typestr=typestr, data=(ptr, False), version=2)


def _in_one_order(lengths, items, supports):
    """Records sorted by a 64-bit key of their items (the same records give the same arrays)."""
    start = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    z = (items.astype(np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    total = np.concatenate([[0], np.cumsum(z ^ (z >> np.uint64(31)), dtype=np.uint64)]).astype(np.uint64)
    order = np.argsort(total[start[1:]] - total[start[:-1]], kind="stable")
    lengths = lengths[order]
    new = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    at = np.arange(new[-1]) - np.repeat(new[:-1] - start[:-1][order], lengths)
    return dict(lengths=lengths.astype(np.int64), items=items[at].astype(np.int64),
                supports=supports[order].astype(np.int64))


def _padded(records, law):
    """Records as int32 arrays of the law's length (longer only where there are more)."""
    sets, items = (1 << 21, 1 << 24) if law == "zipf" else (1 << 17, 1 << 19)
    room = dict(lengths=sets, items=items, supports=sets)
    return {k: np.pad(v.astype(np.int32), (0, max(0, room[k] - len(v))), constant_values=-1) for k, v in records.items()}


class Read(dict):
    """What a call left, as the arrays that make(...) gives of it when it is read."""

    def __init__(self, keys, make, *what):
        super().__init__(dict.fromkeys(keys))
        self.make, self.what, self.read = make, what, None

    def __getitem__(self, key):
        if self.read is None:
            self.read = self.make(*self.what)
        return self.read[key]


def _records(r, law):
    if r.on_device:
        off = _host(r.device_ptrs[0], r.n_sets + 1, "<i8")
        items, supports = _host(r.device_ptrs[1], int(off[-1]), "<i4"), _host(r.device_ptrs[2], r.n_sets, "<i4")
    else:
        off, items, supports = r.set_offsets.astype(np.int64), r.set_items, r.supports
    return _padded(_in_one_order(np.diff(off), items, supports), law)


def Records(result, law):
    return Read(("lengths", "items", "supports"), _records, result, law)


def _classes(costs, order, N):
    return dict(costs=np.pad(costs, (0, N - len(costs))),
                order=np.pad(order.astype(np.int32), (0, N - len(order)), constant_values=-1))


def _host(ptr, n, typestr):
    if n == 0:
        return np.zeros(0, dtype=typestr)
    return torch.as_tensor(_DeviceArray(ptr, n, typestr), device="cuda").cpu().numpy()


def _pairs_in_one_order(p, s, room):
    order = np.lexsort((p[:, 1], p[:, 0]))
    return dict(pairs=np.pad(p[order].astype(np.int32), ((0, room - len(p)), (0, 0)), constant_values=-1),
                supports=np.pad(s[order].astype(np.int32), (0, room - len(s)), constant_values=-1))


def _pairs(n, pairs, supports):
    return _pairs_in_one_order(pairs[:n].cpu().numpy(), supports[:n].cpu().numpy(), len(supports))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "step":
        pre = state["minsup"] if case["prefilter"] else 0
        if case["host"]:
            db = fim.build_vertical_db(state["off"], state["items"], case["N"], word_bits=case["word_bits"],
                                       prefilter_minsup=pre)
        else:
            db = fim.build_vertical_db_device(state["off"], state["items"], case["D"], case["N"],
                                              word_bits=case["word_bits"], prefilter_minsup=pre)
        est = db.estimate_class_costs(SAMPLE_RATE, case["rel"], seed=1, outputs=case["costs"])
        out = dict(found=Records(db.mine(state["minsup"], stats=False), case["law"]))
        if est is not None:
            out["classes"] = Read(("costs", "order"), _classes, *est, case["N"])
        db.free()
        return out
    if kind == "mine":
        return Records(state["db"].mine(state["minsup"], output=case["output"], result_on_device=case["on_device"],
                                        stats=False), case["law"])
    if kind == "plan":
        state["plan"].launch()
        return Records(state["plan"].result(), case["law"])
    if kind == "extend":
        return state["db"].extension_supports(state["prefix"], state["candidates"]).astype(np.int32)
    if kind == "pairs":
        n = state["db"].mine_pairs_noalloc(state["minsup"], state["pairs"], state["supports"], len(state["supports"]))
        return Read(("pairs", "supports"), _pairs, n, state["pairs"], state["supports"])
    ids = [state["server"].submit(off, items, N, minsup, SAMPLE_RATE) for off, items, N, minsup in state["jobs"]]
    out = []
    for i in ids:
        try:
            out.append(Records(state["server"].wait(i)[0], "uniform"))
        except fim.FimError as e:  # a job past its itemset limit
            if e.status != fim.FIM_ERR_OUTPUT_OVERFLOW:
                raise
            out.append(-1)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how far two right answers may differ


def work(case):
    """The database read once (4 bytes per transaction and item) and the answer written; a query reads its
    candidates' bitmap rows instead.  Counting is integer work: AND and popcount, no multiply-adds are needed."""
    if case["kind"] == "serve":
        D = (case["D_hi"] - case["D_lo"]) / math.log(case["D_hi"] / case["D_lo"])
        return dict(bytes=case["jobs"] * D * 4.0 * (1 + 17.5), flops=0)
    if case["kind"] == "extend":
        return dict(bytes=case["D"] / 8.0 * (case["candidates"] + case["prefix"]) + 8.0 * case["candidates"], flops=0)
    return dict(bytes=4.0 * case["D"] * (1 + case["TL"]), flops=0)


def tolerance(case):
    return "exact"  # itemsets, supports and orders are whole numbers; a cost is one division of two of them


def exact(case, seed):
    """Supports by definition, from the transactions as plain numpy and torch count them, where that is quick."""
    kind = case["kind"]
    if kind == "extend":
        off, items = _strata(case, seed)
        x = items.cpu().numpy().reshape(case["D"], int(case["TL"]))
        rng = np.random.RandomState(seed % (1 << 31))
        has = np.ones(case["D"], bool)
        for p in [0] + [int(v) for v in x[0, 1:case["prefix"]]]:
            has &= (x == p).any(1)
        cand = np.sort(rng.permutation(case["N"])[: case["candidates"]])
        return np.bincount(x[has].reshape(-1), minlength=case["N"])[cand].astype(np.int32)
    if kind == "serve" or case["D"] * case["N"] > 1.1e8 or case.get("output", "all") != "all":
        return None
    off, items = _database(case, seed)
    minsup = _minsup(case)
    m = np.zeros((case["N"], case["D"]), bool)
    m[items, np.repeat(np.arange(case["D"]), np.diff(off.astype(np.int64)))] = True
    rows = np.packbits(m, axis=1)
    supp = m.sum(1)
    keep = np.nonzero(supp >= minsup)[0]
    sets, supports = [(int(i),) for i in keep], [int(supp[i]) for i in keep]

    def grow(prefix, bits, later):
        if not len(later):
            return
        both = rows[later] & bits
        c = np.bitwise_count(both).sum(1, dtype=np.int64)
        ok = np.nonzero(c >= minsup)[0]
        for a in ok:
            sets.append(prefix + (int(later[a]),))
            supports.append(int(c[a]))
        if kind == "pairs":
            return
        for n, a in enumerate(ok[:-1]):
            grow(prefix + (int(later[a]),), both[a], later[ok[n + 1:]])

    for n, i in enumerate(keep):
        grow((int(i),), rows[i], keep[n + 1:])
    if kind == "pairs":
        two = [(k, s) for k, s in zip(sets, supports) if len(k) == 2]
        return _pairs_in_one_order(np.array([k for k, _ in two], np.int64).reshape(-1, 2),
                                   np.array([s for _, s in two], np.int64), case["N"] * (case["N"] - 1) // 2)
    lengths = np.array([len(k) for k in sets], np.int64)
    found = _padded(_in_one_order(lengths, np.array([v for k in sets for v in k], np.uint32),
                                  np.array(supports, np.int64)), case["law"])
    return dict(found=found) if kind == "step" else found
