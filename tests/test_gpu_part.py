"""Maps staged in shared memory in part: the plan on both sides of its limits, beside another staged table, and the results."""
import pytest
import torch

from datagen import UNIFORM_I32
from datagen.workloads import AggExpr, ColSpec, DimSpec, KeyExpr, Term, Workload

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None


def _run(n, groups, maps, hashed=True):
    """maps: (keys, largest payload) of each join, every key of a map in use and a few keys beyond it."""
    rand = torch.Generator(device="cuda").manual_seed(n + groups)

    def ints(lo, hi, size):
        return torch.randint(lo, hi, (size,), dtype=torch.int32, device="cuda", generator=rand)

    names = ["fk%d" % i for i in range(len(maps))]
    fact = {"g": ints(0, 2**30, n)}
    dims, specs, value, hit = {}, [], torch.zeros(n, dtype=torch.int64, device="cuda"), None
    for name, (keys, largest) in zip(names, maps):
        dims[name] = {"k": torch.arange(5, keys + 5, dtype=torch.int32, device="cuda"), "v": ints(0, largest + 1, keys)}
        fact[name] = ints(5, keys + 5, n)
        fact[name][:6] = torch.tensor([4, 5, keys + 4, keys + 5, -2**31, 2**31 - 1], dtype=torch.int32)
        specs.append(DimSpec(name, keys, (ColSpec("k", UNIFORM_I32), ColSpec("v", UNIFORM_I32)), key="k", payloads=("v",)))
        at = fact[name].long() - 5
        inside = (at >= 0) & (at < keys)
        hit = inside if hit is None else hit & inside
        value += dims[name]["v"][at.clamp(0, keys - 1)]
    x = Term("PAYLOAD", 0, 0)
    agg = AggExpr("ADD", x, Term("PAYLOAD", 1, 0)) if len(maps) > 1 else AggExpr("COL", x)
    w = Workload("part", n, tuple(ColSpec(c, UNIFORM_I32) for c in fact), tuple(specs), tuple((c, c) for c in names), (),
                 KeyExpr((Term("FACT", "g"),), modulo=groups), agg, "HASHED" if hashed else "DENSE", num_groups=groups,
                 capacity=2 * groups)
    res = sjq.run_workload(w, fact, sjq.build_workload_tables(w, dims), sjq.RunOpts(specialise=True))
    assert res.status() == 0
    g = fact["g"].long()[hit] % groups
    sums = torch.zeros(groups, dtype=torch.int64, device="cuda").index_add_(0, g, value[hit])
    counts = torch.zeros_like(sums).index_add_(0, g, torch.ones_like(g))
    if hashed:
        k, s, c = res.hashed_sorted()
        there = counts.nonzero()[:, 0]
        assert torch.equal(k, there) and torch.equal(s, sums[there]) and torch.equal(c, counts[there])
    else:
        assert torch.equal(res.sums, sums) and torch.equal(res.counts, counts)
    return res.info.describe()


ROWS = 2**24 + 3


@pytest.mark.parametrize("keys,largest,groups,hashed,staged", [
    (700_000, 3, 1_000_000, True, 1),    # 175 KB, whole
    (800_000, 3, 1_000_000, True, 0),    # 200 KB: left to the L1
    (800_000, 3, 20_000, True, 2),       # (of few groups, and of a dense result, the first 192 KB)
    (800_000, 3, 200_000, False, 2),
    (880_000, 3, 1_000_000, True, 0),    # 215 KB
    (890_000, 3, 1_000_000, True, 2),
    (250_000, 200, 1_000_000, True, 0),  # 250 KB, codes of a byte
    (350_000, 200, 1_000_000, True, 2),
    (4_700_000, 3, 1_000_000, True, 2),  # 1,148 KB
    (4_750_000, 3, 1_000_000, True, 0),  # 1,160 KB: too little of it
    (4_750_000, 3, 200_000, True, 2),
    (2_000_000, 3, 2_097_152, True, 2),  # the largest group table
    (2_000_000, 3, 2_097_153, True, 0),
])
def test_the_part_of_a_map_that_is_staged(keys, largest, groups, hashed, staged):
    plan = _run(ROWS, groups, [(keys, largest)], hashed)
    assert plan["agg_path"] == "global" and plan["in_smem"][0] == staged
    assert plan["block"] == (768 if staged else 384)


@pytest.mark.parametrize("first", [2_556, 40_000, 120_000])
@pytest.mark.parametrize("keys,largest", [(300_000, 3), (3_000_000, 3)])
def test_a_part_beside_another_staged_map_stays_within_the_carve_out(first, keys, largest):
    plan = _run(ROWS, 100_000, [(first, 3), (keys, largest)])
    assert sorted(plan["in_smem"][:2]) == [1, 1 if keys == 300_000 else 2]
    assert plan["smem_bytes"] <= 196 * 1024 - 1024 - 512 and plan["block"] == 768


@pytest.mark.parametrize("keys,largest,block", [(1_500_000, 3, 768), (2_000_000, 3, 512), (3_100_000, 3, 512),
                                                (3_200_000, 3, 768), (500_000, 200, 768)])
def test_block_sizes_of_many_rows(keys, largest, block):
    plan = _run(2**26 + 1, 50_000, [(keys, largest)])
    assert plan["in_smem"][0] == 2 and plan["block"] == block
