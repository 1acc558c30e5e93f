"""Runs, lists, sorts, merges and chunked host runs inside CUDA graphs: the kernels are launched while their predecessors
still run (programmatic edges of the graph), and a replay sees the data of the moment."""
import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, KeyExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, oracle_result, to_dev  # noqa: E402
from qhelpers import adhoc  # noqa: E402


def _data(n, groups, seed):
    rng = np.random.default_rng(seed)
    return {"p": rng.integers(0, 1000, n).astype(np.int32), "g": rng.integers(0, groups, n).astype(np.int32),
            "m": rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)}


@pytest.mark.parametrize("mode,groups,modulo", [("SCALAR", 1, 0), ("DENSE", 500, 0), ("DENSE", 100_000, 0),
                                                ("HASHED", 500, 500), ("HASHED", 30_000, 30_000), ("HASHED", 5_000, 0)])
@pytest.mark.parametrize("compiled", [False, True])
def test_a_captured_run_and_sort_replay_on_new_data(mode, groups, modulo, compiled):
    n = 600_011
    key = None if mode == "SCALAR" else KeyExpr((Term("FACT", "g"),), offset=0, modulo=modulo)
    first = _data(n, groups, 1)
    w = adhoc("captured", first, [], [], [Pred("p", "LT", 300)], key, AggExpr("COL", Term("FACT", "m")), mode,
              num_groups=groups, capacity=groups + 8)
    fact, opts = to_dev(first), sjq.RunOpts(specialise=compiled)
    res = sjq.run_workload(w, fact, {}, opts)  # modules are compiled and loaded outside the capture
    if mode == "HASHED":
        res.sort()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sjq.run_workload(w, fact, {}, opts, result=res)
        if mode == "HASHED":
            res.sort()
    for seed in (2, 3):
        data = _data(n, groups, seed)
        for c, v in data.items():
            fact[c].copy_(torch.from_numpy(v))
        graph.replay()
        torch.cuda.synchronize()
        assert res.status() == 0
        exp = oracle_result(w, data, {})[1]
        if mode == "HASHED":  # in order already
            k = int(res.n_groups.item())
            assert np.array_equal(res.keys[:k].cpu().numpy(), exp["keys"])
        compare(w, res, exp)


def test_a_captured_merge_and_a_captured_host_run():
    n = 300_007
    w = adhoc("captured", _data(n, 400, 1), [], [], [Pred("p", "LT", 300)], KeyExpr((Term("FACT", "g"),), modulo=400),
              AggExpr("COL", Term("FACT", "m")), "HASHED", capacity=500)
    pinned = {c: torch.from_numpy(v).pin_memory() for c, v in _data(n, 400, 1).items()}
    staging = torch.empty(sjq.staging_bytes(pinned, 65_536), dtype=torch.uint8, device="cuda")
    lists = [torch.zeros(800, dtype=torch.int64, device="cuda") for _ in range(3)]
    res, host = sjq.run_workload_host(w, pinned, {}, staging, 65_536)
    merged = sjq.merge_groups(*lists, 500)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sjq.run_workload_host(w, pinned, {}, staging, 65_536, result=res, host=host)
        for part, whole in zip(lists, (res.keys, res.sums, res.counts)):
            part[:400].copy_(whole[:400])  # every group occurs
            part[400:].copy_(whole[:400])
        sjq.merge_groups(*lists, 500, result=merged)
    data = _data(n, 400, 5)
    for c, v in data.items():
        pinned[c].copy_(torch.from_numpy(v))
    graph.replay()
    torch.cuda.synchronize()
    exp = oracle_result(w, data, {})[1]
    compare(w, res, exp)
    assert len(exp["keys"]) == 400 and merged.status() == 0
    k, s, c = (t.cpu().numpy() for t in merged.hashed_sorted())
    with np.errstate(over="ignore"):
        assert np.array_equal(k, exp["keys"]) and np.array_equal(s, 2 * exp["sums"]) and np.array_equal(c, 2 * exp["counts"])
