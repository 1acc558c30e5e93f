"""Hashed group-bys at the sizes where their table, its listing and the adds into it change form: part of a warp, one
tile and one more, several tiles per block; groups indexed by the key and groups in the hash table; few and all rows
surviving; capacity reached and exceeded."""
import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, KeyExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, run_both  # noqa: E402
from qhelpers import adhoc  # noqa: E402


def _query(n, groups, below, capacity, modulo, seed=1):
    rng = np.random.default_rng(seed)
    fact = {"p": rng.integers(0, 1000, n).astype(np.int32), "g": rng.integers(0, groups, n).astype(np.int32),
            "m": rng.integers(-2**31, 2**31 - 1, n).astype(np.int32)}
    fact["g"][:groups] = np.arange(min(n, groups))  # every group occurs
    return fact, adhoc("hashed", fact, [], [], [Pred("p", "LT", below)],
                       KeyExpr((Term("FACT", "g"),), offset=0, modulo=modulo), AggExpr("COL", Term("FACT", "m")),
                       "HASHED", capacity=capacity)


@pytest.mark.parametrize("n,groups", [(1, 1), (31, 7), (33, 33), (5_000, 2047), (5_000, 2048), (5_000, 2049),
                                      (50_000, 1024), (400_003, 150_001)])
@pytest.mark.parametrize("below", [1000, 10])
def test_lists_of_every_length(n, groups, below):
    for modulo in (groups, 0):  # indexed by the key, in the hash table
        fact, w = _query(n, groups, below, max(8, groups), modulo)
        for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True), sjq.RunOpts(group_hash_always=True),
                     sjq.RunOpts(specialise=True, compaction=1), sjq.RunOpts(specialise=True, pass_ppm=[below * 1000])):
            res, exp, _ = run_both(w, fact, {}, opts=opts)
            assert res.status() == 0
            compare(w, res, exp)


@pytest.mark.parametrize("groups", [1, 2, 1024, 1025, 4096, 4097, 20_000])
@pytest.mark.parametrize("below", [1000, 10])
def test_an_indexed_table_is_listed_in_key_order_by_one_kernel_where_it_is_small(groups, below):
    """2 M - 1 cells: up to four blocks of 2048 count the groups before their own themselves."""
    fact, w = _query(60_001, groups, below, groups + 8, groups)
    for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True)):
        res, exp, _ = run_both(w, fact, {}, opts=opts)
        assert res.status() == 0 and res.info.kernel_launches == (3 if groups <= 4096 else 4)
        n = int(res.n_groups.item())
        assert np.array_equal(res.keys[:n].cpu().numpy(), exp["keys"])  # as listed, not sorted
        assert np.array_equal(res.sums[:n].cpu().numpy(), exp["sums"])
        compare(w, res, exp)


def test_large_indexed_table_has_several_tiles_per_block():
    fact, w = _query(200_003, 150_000, 1000, 3_000_000, 5_000_000)  # ten million cells, 2048 to a tile
    res, exp, _ = run_both(w, fact, {}, opts=sjq.RunOpts(specialise=True))
    assert res.status() == 0
    compare(w, res, exp)


def test_capacity_is_a_limit_in_both_forms():
    for modulo in (100, 0):
        fact, w = _query(10_000, 100, 1000, 99, modulo)
        for opts in (sjq.RunOpts(), sjq.RunOpts(specialise=True)):
            res, _, _ = run_both(w, fact, {}, opts=opts, check=False)
            assert res.status() == 19


@pytest.mark.parametrize("n", [1, 31, 33, 100_003, 303_103, 303_105, 1_000_003])
def test_merge_adds_zero_and_wrapping_entries(n):
    rng = np.random.default_rng(n)
    keys = rng.integers(-5, max(6, n // 3), n)
    keys[0] = np.iinfo(np.int64).min  # the empty marker is a legal key
    sums, counts = rng.integers(-2**63, 2**63 - 1, n), rng.integers(0, 2, n)
    counts[0] = 1
    res = sjq.merge_groups(*(torch.from_numpy(a.astype(np.int64)).cuda() for a in (keys, sums, counts)), n)
    assert res.status() == 0
    k, s, c = (t.cpu().numpy() for t in res.hashed_sorted())
    want, inverse = np.unique(keys, return_inverse=True)
    ws, wc = np.zeros(len(want), np.int64), np.zeros(len(want), np.int64)
    with np.errstate(over="ignore"):
        np.add.at(ws, inverse, sums)
    np.add.at(wc, inverse, counts)
    assert np.array_equal(k, want) and np.array_equal(s, ws) and np.array_equal(c, wc)
