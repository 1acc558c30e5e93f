"""Results that the pass clears itself, at the sizes where the clear's shares and the launch change; and the forms of the
ahead-of-time kernels (queues or none, 32-bit codes or any) on both sides of the rule that picks them."""
import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, KeyExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, oracle_result, run_both, to_dev  # noqa: E402
from qhelpers import adhoc  # noqa: E402


def _grouped(n, groups, seed):
    rng = np.random.default_rng(seed)
    return {"p": rng.integers(0, 1000, n).astype(np.int32), "g": rng.integers(0, groups, n).astype(np.int32),
            "m": rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)}


def _query(fact, groups):
    key = None if groups == 0 else KeyExpr((Term("FACT", "g"),))
    return adhoc("cleared", fact, [], [], [Pred("p", "LT", 300)], key, AggExpr("COL", Term("FACT", "m")),
                 "SCALAR" if groups == 0 else "DENSE", num_groups=max(1, groups))


@pytest.mark.parametrize("n", [1, 1537, 2**19, 2**19 + 1])
@pytest.mark.parametrize("groups", [0, 1, 2, 767, 769, 4_096, 4_097])
@pytest.mark.parametrize("compiled", [False, True])
def test_small_results_are_cleared_by_their_pass(n, groups, compiled):
    """Buffers and words full of what earlier runs left: one launch clears and fills them, again and again, and leaves the
    words at zero; without the words, or beyond the limits, a kernel before the pass does."""
    opts = sjq.RunOpts(specialise=compiled, agg_path=1 if 1 < groups <= 4_096 else 0)  # the largest shared table
    fact = _grouped(n, max(1, groups), n + groups)
    w = _query(fact, groups)
    res, exp, _ = run_both(w, fact, {}, opts)
    dev = to_dev(fact)
    by_pass = n <= 2**19 and groups <= 4_096
    for words in (torch.full((8,), -1, dtype=torch.int64, device="cuda"), torch.zeros(8, dtype=torch.int64, device="cuda"), None):
        res.sync = words
        for _ in range(3):
            for t in (res.sums, res.counts, res.status_dev):
                t.fill_(77)
            sjq.run_workload(w, dev, {}, opts, result=res)
        assert res.status() == 0 and res.info.kernel_launches == (1 if by_pass and words is not None else 2)
        compare(w, res, exp)
        if by_pass and words is not None:
            assert words[0] == 0 and ((words == 0) | (words == -1)).all()  # (as many flags as blocks that clear)
    res.sync = torch.full((8,), 5, dtype=torch.int64, device="cuda")  # a run that accumulates clears nothing
    opts.accumulate = True
    sjq.run_workload(w, dev, {}, opts, result=res)
    torch.cuda.synchronize()
    assert (res.sync == 5).all()
    compare(w, res, {k: (2 * v if k in ("sum", "count", "sums", "counts") else v) for k, v in exp.items()})


@pytest.mark.parametrize("groups,limit", [(100, 99), (500, 1)])  # shared table, registers
def test_a_key_out_of_range_is_told_by_a_pass_that_clears(groups, limit):
    fact = _grouped(40_001, groups, 3)
    fact["g"][:groups] = np.arange(groups)
    fact["p"][:groups] = 0
    w = _query(fact, limit)
    for _ in range(2):
        res = sjq.run_workload(w, to_dev(fact), {})
        assert res.info.kernel_launches == 1 and res.status() == 18  # SJQ_ERR_GROUP_RANGE
    fact["g"] %= limit  # ... and forgotten by the next one
    sjq.run_workload(w, to_dev(fact), {}, result=res)
    assert res.status() == 0
    compare(w, res, oracle_result(w, fact, {})[1])


@pytest.mark.parametrize("groups", [0, 20])
@pytest.mark.parametrize("compiled", [False, True])
def test_a_captured_pass_that_clears_replays_on_new_data(groups, compiled):
    n, opts = 100_003, sjq.RunOpts(specialise=compiled)
    first = _grouped(n, max(1, groups), 1)
    w, fact = _query(first, groups), to_dev(first)
    res = sjq.run_workload(w, fact, {}, opts)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sjq.run_workload(w, fact, {}, opts, result=res)
    assert res.info.kernel_launches == 1
    for seed in (2, 3, 4):
        data = _grouped(n, max(1, groups), seed)
        for c, v in data.items():
            fact[c].copy_(torch.from_numpy(v))
        graph.replay()
        torch.cuda.synchronize()
        assert res.status() == 0
        compare(w, res, oracle_result(w, data, {})[1])


@pytest.mark.parametrize("n", [5, 70_001, 600_011])  # without and with queues
@pytest.mark.parametrize("key64", [False, True])
@pytest.mark.parametrize("payloads", [(), ("a",), ("a", "b"), ("wide",)])
@pytest.mark.parametrize("mult", [1, 2**33])
@pytest.mark.parametrize("hashed", [False, True])
def test_forms_by_key_code_and_multiplier(n, key64, payloads, mult, hashed):
    """Codes of no, 32 and 64 bits behind 32- and 64-bit keys, contributions within and beyond 32 bits, 64-bit measures."""
    rng = np.random.default_rng(n + len(payloads))
    rows = 3_000
    keys = rng.permutation(rows * 3)[:rows].astype(np.int64 if key64 else np.int32) - rows
    dim = {"k": keys, "a": rng.integers(-9, 9, rows).astype(np.int32), "b": rng.integers(0, 2**20, rows).astype(np.int32),
           "wide": rng.integers(-2**50, 2**50, rows), "f": rng.integers(0, 4, rows).astype(np.int32)}
    fact = {"fk": rng.integers(-rows, 2 * rows, n).astype(keys.dtype), "m": rng.integers(-2**31, 2**31 - 1, n).astype(np.int32),
            "l": rng.integers(-2**62, 2**62, n), "g": rng.integers(0, 40, n).astype(np.int32)}
    for measure in ("m", "l"):
        x = Term("PAYLOAD", 0, len(payloads) - 1, mult) if payloads else Term("FACT", measure, 0, mult)
        w = adhoc("forms", fact, [("d", dim, "k", [Pred("f", "LT", 2)], list(payloads), hashed)], [("fk", "d")],
                  [Pred("g", "LT", 35)], KeyExpr((Term("FACT", "g"),)), AggExpr("ADD", x, Term("FACT", measure)), "DENSE",
                  num_groups=40)
        res, exp, _ = run_both(w, fact, {"d": dim})
        assert res.status() == 0
        compare(w, res, exp)


@pytest.mark.parametrize("keys", [200_000, 786_431, 786_432, 786_433, 1_600_000])  # 2-bit codes: 192 KB hold 786,432
@pytest.mark.parametrize("payload", [3, 200])
@pytest.mark.parametrize("hashed", [False, True])
def test_a_map_staged_whole_and_in_part(keys, payload, hashed):
    """2- and 8-bit codes on both sides of what is staged; keys below, on the edges of and beyond the map's range."""
    n, rng = 2**24 + 3, np.random.default_rng(keys)
    dim = {"k": np.arange(7, keys + 7, dtype=np.int32), "v": rng.integers(0, payload + 1, keys).astype(np.int32)}
    fact = {"fk": rng.integers(5, keys + 9, n).astype(np.int32), "g": rng.integers(0, 2**30, n).astype(np.int32)}
    edges = np.array([6, 7, 7 + 196_607, 7 + 196_608, 7 + 786_431, 7 + 786_432, 6 + keys, 7 + keys, -2**31, 2**31 - 1])
    fact["fk"][:10] = edges
    groups = 50_000
    w = adhoc("part", fact, [("d", dim, "k", [], ["v"])], [("fk", "d")], [], KeyExpr((Term("FACT", "g"),), modulo=groups),
              AggExpr("ADD", Term("FACT", "fk"), Term("PAYLOAD", 0, 0)), "HASHED" if hashed else "DENSE", num_groups=groups,
              capacity=2 * groups)
    opts = sjq.RunOpts(specialise=True)
    tables = sjq.build_workload_tables(w, {"d": to_dev(dim)})
    dev = to_dev(fact)
    res = sjq.run_workload(w, dev, tables, opts)
    assert res.status() == 0 and res.info.describe()["in_smem"][0] == (1 if keys * (2 if payload == 3 else 8) < 8 * 192 * 1024 else 2)
    hit = (fact["fk"] >= 7) & (fact["fk"] < keys + 7)
    at, g = fact["fk"][hit].astype(np.int64), fact["g"][hit] % groups
    value = at + dim["v"][at - 7]
    sums = np.bincount(g, weights=value.astype(np.float64), minlength=groups)  # below 2**53: exact
    counts = np.bincount(g, minlength=groups)
    k, s, c = res.hashed_sorted() if hashed else (None, res.sums, res.counts)
    assert hashed is False or np.array_equal(k.cpu().numpy(), np.arange(groups))
    assert np.array_equal(s.cpu().numpy(), sums.astype(np.int64)) and np.array_equal(c.cpu().numpy(), counts)
