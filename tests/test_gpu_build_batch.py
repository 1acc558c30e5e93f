"""Open-addressing tables of several forms built in one batch, at sizes where a warp's lanes take key after key."""
import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, run_both  # noqa: E402
from qhelpers import adhoc  # noqa: E402

FORMS = {"none": [], "usual": ["a"], "wide": ["w"], "two": ["a", "b"]}


@pytest.mark.parametrize("rows", [129, 4_099, 60_013, 400_001])
@pytest.mark.parametrize("forms", [("usual", "wide"), ("none", "two"), ("wide", "usual", "none", "two"), ("usual", "none")])
@pytest.mark.parametrize("key64", [False, True])
@pytest.mark.parametrize("kept", [1, 8])  # of eight rows
def test_batches_of_several_forms(rows, forms, key64, kept):
    rng = np.random.default_rng(rows + len(forms))
    ktype = np.int64 if key64 else np.int32
    dims, fact, specs, joins = {}, {}, [], []
    n = 50_003
    for i, form in enumerate(forms):
        m = rows - 7 * i  # (the dimensions of a batch do not end together)
        keys = rng.permutation(3 * m)[:m].astype(ktype)
        if key64:
            keys = keys * 0x9E3779B97F4A7 - 2**61
        name = "d%d" % i
        dims[name] = {"k": keys, "f": rng.integers(0, 8, m).astype(np.int32), "a": rng.integers(-9, 2**20, m).astype(np.int32),
                      "b": rng.integers(0, 40, m).astype(np.int32), "w": rng.integers(-2**50, 2**50, m)}
        specs.append((name, dims[name], "k", [Pred("f", "LT", kept)], FORMS[form], True))
        fact["fk%d" % i] = np.where(rng.random(n) < 0.95, keys[rng.integers(0, m, n)], ktype(1))
        joins.append(("fk%d" % i, name))
    fact["m"] = rng.integers(0, 1000, n).astype(np.int32)
    for i, form in enumerate(forms):  # the payloads of each dimension in turn
        for p in range(len(FORMS[form])):
            w = adhoc("batch", fact, specs, joins, [], None, AggExpr("ADD", Term("FACT", "m"), Term("PAYLOAD", i, p)), "SCALAR")
            res, exp, tables = run_both(w, fact, dims)
            assert res.status() == 0
            assert [sjq.build_launches(t) for t in tables.values()] == [3] + [0] * (len(forms) - 1)
            compare(w, res, exp)
