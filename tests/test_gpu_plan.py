"""The evaluation order the planner chooses, and parity where its search changes form."""
import ctypes

import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, KeyExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, oracle_result, run_both, to_dev  # noqa: E402
from qhelpers import adhoc  # noqa: E402


@pytest.mark.parametrize("small_first", [True, False])
def test_of_two_equally_selective_joins_the_one_in_shared_memory_goes_first(small_first):
    n, rng = 50_003, np.random.default_rng(3)
    sizes = {"small": 100_000, "large": 1_000_000}  # bitmaps of 12 KB and 125 KB
    dims = [(nm, {"k": np.arange(rows, dtype=np.int32), "a": (np.arange(rows) % 25).astype(np.int32)}, "k",
             [Pred("a", "EQ", 7)], []) for nm, rows in sizes.items()]
    fact = {nm: rng.integers(0, rows, n).astype(np.int32) for nm, rows in sizes.items()}
    fact["m"] = rng.integers(0, 1000, n).astype(np.int32)
    names = list(sizes) if small_first else list(sizes)[::-1]
    w = adhoc("order", fact, dims, [(nm, nm) for nm in names], [], None, AggExpr("COL", Term("FACT", "m")), "SCALAR")
    res, exp, _ = run_both(w, fact, {d[0]: d[1] for d in dims})
    compare(w, res, exp)
    assert res.info.order[0] == names.index("small")


@pytest.mark.parametrize("npreds", [1, 8, 9, 10, 11, 12, 16])
def test_any_number_of_filters(npreds):
    n, rng = 20_011, np.random.default_rng(npreds)
    fact = {f"c{i}": rng.integers(0, 100, n).astype(np.int32) for i in range(npreds)}
    dim = {"k": np.arange(100, dtype=np.int32), "a": (np.arange(100) % 2).astype(np.int32)}
    w = adhoc("many", fact, [("d", dim, "k", [Pred("a", "EQ", 1)], [])], [("c0", "d")],
              [Pred(f"c{i}", "LT", 80 + i) for i in range(npreds)], None, AggExpr("COL", Term("FACT", "c0")), "SCALAR")
    for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True)):
        res, exp, _ = run_both(w, fact, {"d": dim}, opts=opts)
        assert res.status() == 0
        compare(w, res, exp)
        assert sorted(res.info.order[: npreds + 1]) == list(range(npreds + 1))


@pytest.mark.parametrize("n", [2**19 - 1, 2**19, 2**19 + 1, 700_001])
@pytest.mark.parametrize("below", [2, 10, 60, 130, 400])
def test_launch_shapes_by_rows_and_survivors(n, below):
    """Queue-free plans up to 2^19 rows, queues beyond; eight or sixteen rows per thread at level 0; a queue for the
    second filter or not."""
    rng = np.random.default_rng(below)
    fact = {"p": rng.integers(0, 1000, n).astype(np.int32), "q": rng.integers(0, 1000, n).astype(np.int32),
            "fk": rng.integers(0, 50_000, n).astype(np.int32), "m": rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)}
    dim = {"k": np.arange(50_000, dtype=np.int32), "a": (np.arange(50_000) % 3).astype(np.int32)}
    preds = [Pred("p", "LT", below), Pred("q", "LT", 300)]
    w = adhoc("shapes", fact, [("d", dim, "k", [Pred("a", "EQ", 1)], [])], [("fk", "d")], preds, None,
              AggExpr("COL", Term("FACT", "m")), "SCALAR")
    ppm = [below * 1000, 300_000]
    for opts in (sjq.RunOpts(pass_ppm=ppm), sjq.RunOpts(specialise=True, pass_ppm=ppm)):
        res, exp, _ = run_both(w, fact, {"d": dim}, opts=opts)
        assert res.status() == 0
        compare(w, res, exp)
        assert (res.info.reserved_levels == 0) == (n <= 2**19)


@pytest.mark.parametrize("shift", [0, 2])
def test_64_bit_columns_on_16_and_32_byte_boundaries(shift):
    """Four 64-bit values are one 256-bit load where the column starts on a 32-byte boundary, else two loads."""
    n, rng = 600_007, np.random.default_rng(8)
    keys = rng.permutation(5_000).astype(np.int64) * 2**33
    dim = {"k": keys, "p": rng.integers(0, 99, 5_000).astype(np.int32)}
    fact = {"fk": rng.choice(np.concatenate([keys, keys + 1]), n), "m": rng.integers(-2**62, 2**62, n)}
    w = adhoc("wide", fact, [("d", dim, "k", [], ["p"], True)], [("fk", "d")], [], KeyExpr((Term("PAYLOAD", 0, 0),)),
              AggExpr("COL", Term("FACT", "m")), "DENSE", num_groups=99)
    dev = {}
    for c, v in fact.items():
        room = torch.empty(n + shift, dtype=torch.int64, device="cuda")
        dev[c] = room[shift:].copy_(torch.from_numpy(v))
        assert dev[c].data_ptr() % 32 == 8 * shift % 32
    tables = None
    for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True), sjq.RunOpts(compaction=1), sjq.RunOpts(specialise=True, compaction=1)):
        res, exp, tables = run_both(w, fact, {"d": dim}, opts=opts, dev_fact=dev, tables=tables)
        assert res.status() == 0
        compare(w, res, exp)


@pytest.mark.parametrize("n", [2**20 - 1, 2**20, 1_300_001])
def test_host_resident_filters_are_ordered_by_the_bus(n):
    """From 2^20 rows on the order copies as few columns as it can: of three filters that keep a fifth, a fifth and a
    third, the first two are copied and the last is read in place; below it is the order of a device-resident run."""
    rng = np.random.default_rng(n)
    dims, fact, host = [], {}, {}
    for nm, rows, of in (("wide", 400_000, 5), ("other", 400_000, 5), ("small", 3_000, 3)):
        host[nm] = {"k": rng.permutation(rows).astype(np.int32), "a": (np.arange(rows) % of).astype(np.int32)}
        dims.append((nm, host[nm], "k", [Pred("a", "EQ", 1)], []))
        fact[nm] = rng.integers(0, rows, n).astype(np.int32)
    fact["m"] = rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)
    w = adhoc("bus", fact, dims, [(d[0], d[0]) for d in dims], [], None, AggExpr("COL", Term("FACT", "m")), "SCALAR")
    _, exp, tables = run_both(w, fact, host)
    pinned = {c: torch.from_numpy(v).pin_memory() for c, v in fact.items()}
    how = {c: h for c, (h, _) in sjq.host_transfer_plan(pinned, (), [(d[0], tables[d[0]]) for d in dims], None, w.agg).items()}
    assert how["small"] == ("in place" if n >= 2**20 else "copy") and how["m"] == "in place"
    for chunk in (2**18, 2**21):
        staging = torch.empty(sjq.staging_bytes(pinned, chunk), dtype=torch.uint8, device="cuda")
        for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True), sjq.RunOpts(host_copy_all=True), sjq.RunOpts(order=(2, 0, 1))):
            res, out = sjq.run_workload_host(w, pinned, tables, staging, chunk, opts)
            torch.cuda.synchronize()
            assert int(out.status[0]) == 0
            compare(w, res, exp)


def _modules():
    """Compiled modules loaded since the last call; all are unloaded (nothing is running)."""
    torch.cuda.synchronize()
    lib = sjq.sjq.lib()
    lib.sjq_jit_cache_clear.restype = ctypes.c_int32
    return lib.sjq_jit_cache_clear()


def _sparse_query(n):
    """Of a thousand rows one passes both filters: q is read for a twentieth of the rows, m for one in a thousand."""
    rng = np.random.default_rng(n)
    fact = {c: rng.integers(0, 1000, n).astype(np.int32) for c in ("p", "q", "m")}
    return fact, adhoc("sparse", fact, [], [], [Pred("p", "LT", 50), Pred("q", "LT", 20)], None,
                       AggExpr("COL", Term("FACT", "m")), "SCALAR")


@pytest.mark.parametrize("n", [100_003, 2**19])
def test_few_rows_with_columns_in_place_are_queued_like_many(n):
    """A kernel without queues would fetch columns in host memory for rows that need none of them: with such a column a
    small table runs through the kernel that a large one does, with copies alone through one without queues."""
    for copy_all, modules in ((False, 1), (True, 2)):
        _modules()
        for rows in (700_001, n):
            fact, w = _sparse_query(rows)
            pinned = {c: torch.from_numpy(v).pin_memory() for c, v in fact.items()}
            opts = sjq.RunOpts(specialise=True, pass_ppm=(50_000, 20_000), host_copy_all=copy_all)
            how = sjq.host_transfer_plan(pinned, w.preds, (), None, w.agg, opts)
            assert how["m"][0] == ("copy" if copy_all else "in place")
            staging = torch.empty(sjq.staging_bytes(pinned, 700_004), dtype=torch.uint8, device="cuda")
            res, out = sjq.run_workload_host(w, pinned, {}, staging, 700_004, opts)
            torch.cuda.synchronize()
            assert int(out.status[0]) == 0
            compare(w, res, oracle_result(w, fact, {})[1])
        assert _modules() == modules


@pytest.mark.parametrize("tail", [4, 50_003, 2**19])
def test_a_short_last_chunk_runs_through_the_kernel_of_the_others(tail):
    """One module for a whole run from host memory: groups, a staged table and columns copied or read in place."""
    chunk = 2**20
    rng = np.random.default_rng(tail)
    dim = {"k": np.arange(3_000, dtype=np.int32), "a": rng.integers(0, 100, 3_000).astype(np.int32)}
    fact, w = _sparse_query(2 * chunk + tail)
    fact["fk"] = rng.integers(0, 3_000, len(fact["p"])).astype(np.int32)
    w = adhoc("tail", fact, [("d", dim, "k", [], ["a"])], [("fk", "d")], w.preds, KeyExpr((Term("PAYLOAD", 0, 0),)),
              AggExpr("COL", Term("FACT", "m")), "DENSE", num_groups=100)
    tables = sjq.build_workload_tables(w, {"d": to_dev(dim)})
    pinned = {c: torch.from_numpy(v).pin_memory() for c, v in fact.items()}
    staging = torch.empty(sjq.staging_bytes(pinned, chunk), dtype=torch.uint8, device="cuda")
    exp = oracle_result(w, fact, {"d": dim})[1]
    for opts in (sjq.RunOpts(specialise=True), sjq.RunOpts(specialise=True, host_copy_all=True)):
        _modules()
        res, out = sjq.run_workload_host(w, pinned, tables, staging, chunk, opts)
        torch.cuda.synchronize()
        assert int(out.status[0]) == 0
        compare(w, res, exp)
        assert _modules() == 1


@pytest.mark.parametrize("n", [20_011, 2**19])
def test_options_for_queues_hold_for_few_rows_too(n):
    """A kernel without queues has no batches of survivors, no level 0 and no staged first column."""
    fact, w = _sparse_query(n)
    for kw, status in ((dict(rows_per_lane=4), 0), (dict(rows_per_lane=8, specialise=True), 0),
                       (dict(dense_slots=4, specialise=True), 0), (dict(l0_bulk=1, specialise=True), 0),
                       (dict(l0_bulk=3, specialise=True, block_threads=128, ctas_per_sm=1), 22)):
        res, exp, _ = run_both(w, fact, {}, opts=sjq.RunOpts(**kw))
        assert res.info.reserved_levels > 0
        assert res.status() == status
        compare(w, res, exp)
    res, exp, _ = run_both(w, fact, {}, opts=sjq.RunOpts(dense_slots=2, rows_per_lane=4, l0_bulk=2, compaction=1))
    assert res.info.reserved_levels == 0
    compare(w, res, exp)
