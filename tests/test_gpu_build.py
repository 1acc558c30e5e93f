"""Table builds at the sizes and key orders where their kernels take another path: parts of a thread's four rows, a
warp's 128, a block's 1024; neighbouring, descending, scattered and widely spaced keys; repeated keys inside a thread,
a warp, a block and across blocks; tables without a presence bitmap; batches of more dimensions and filters than one
launch takes."""
import threading

import numpy as np
import pytest
import torch

from datagen.workloads import AggExpr, KeyExpr, Pred, Term

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, run_both, to_dev  # noqa: E402
from qhelpers import adhoc  # noqa: E402

SIZES = [1, 3, 4, 5, 127, 128, 129, 1023, 1024, 1025, 40_961]


def _keys(n, order, wide, rng):
    k = np.arange(n, dtype=np.int64)
    if order == "descending":
        k = k[::-1].copy()
    elif order == "scattered":
        k = rng.permutation(n)
    elif order == "spaced":
        k = k * 37
    k = k - n // 2
    return k if wide else k.astype(np.int32)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("order", ["ascending", "descending", "scattered", "spaced"])
def test_tables_of_every_form(n, order):
    rng = np.random.default_rng(n)
    for wide in (False, True):
        keys = _keys(n, order, wide, rng)
        for span, forced in ((0, False), (3, False), (13, False), (200, False), (40_000, False), (2**31 - 1, False),
                             (2**40, False), (0, True), (1000, True), (2**40, True)):
            dim = {"k": keys, "f": rng.integers(0, 3, n).astype(np.int32)}
            pay = []
            if span:
                dim["p"] = rng.integers(0, span, n, endpoint=True).astype(np.int64 if span > 2**31 else np.int32)
                pay = ["p"]
            fk = rng.integers(int(keys.min()) - 5, int(keys.max()) + 6, 3 * n + 7)
            fact = {"fk": fk.astype(keys.dtype), "m": rng.integers(0, 1000, len(fk)).astype(np.int32)}
            agg = AggExpr("ADD", Term("FACT", "m"), Term("PAYLOAD", 0, 0)) if pay else AggExpr("COL", Term("FACT", "m"))
            w = adhoc("forms", fact, [("d", dim, "k", [Pred("f", "NE", 1)], pay, forced)], [("fk", "d")], [], None, agg,
                      "SCALAR")
            res, exp, _ = run_both(w, fact, {"d": dim})
            assert res.status() == 0
            compare(w, res, exp)


@pytest.mark.parametrize("apart", [1, 3, 40, 500, 30_000])
@pytest.mark.parametrize("order", ["ascending", "scattered"])
def test_a_repeated_key_is_found_wherever_its_rows_are(apart, order):
    n, rng = 40_000, np.random.default_rng(apart)
    keys = _keys(n, order, False, rng)
    at = 5_001
    keys[at + apart] = keys[at]
    for pay_max, forced in ((0, False), (13, False), (200, False), (40_000, False), (2**31 - 1, False), (1000, True)):
        cols = {"k": keys, "p": np.full(n, pay_max, np.int32)}
        cols["p"][0] = 0
        dev = to_dev(cols)
        pay = ("p",) if pay_max else ()
        assert sjq.build_dim(dev, "k", (), pay, force_kind=sjq.sjq.FORCE_HASH if forced else 0).status() == 16
        if pay_max >= 200 and not forced:  # codes of a byte and more may do without the bitmap
            def bare(L):
                L.filter_bits = 0
                L.table_bytes = sjq.layout_bytes(L)

            assert sjq.build_dim(dev, "k", (), pay, edit_layout=bare).status() == 16
            keep = np.delete(np.arange(n), at + apart)
            t = sjq.build_dim(to_dev({c: v[keep] for c, v in cols.items()}), "k", (), pay, edit_layout=bare)
            assert t.status() == 0


def test_more_dimensions_and_filters_than_one_launch_takes():
    rng = np.random.default_rng(5)
    n, fact, dims, joins, host = 30_011, {}, [], [], {}
    for j in range(8):
        rows = [2_500, 1, 1024, 70_000, 33, 5_000, 128, 10][j]
        dim = {"k": rng.permutation(rows).astype(np.int32)}
        preds = []
        for f in range(j + 1):
            dim[f"f{f}"] = rng.integers(0, 100, rows).astype(np.int32)
            preds.append(Pred(f"f{f}", "GE", 1))
        dim["p"] = rng.integers(0, 50, rows).astype(np.int32)
        fact[f"fk{j}"] = rng.integers(0, rows, n).astype(np.int32)
        dims.append((f"d{j}", dim, "k", preds, ["p"]))
        joins.append((f"fk{j}", f"d{j}"))
        host[f"d{j}"] = dim
    w = adhoc("eight", fact, dims, joins, [], KeyExpr((Term("PAYLOAD", 0, 0),)),
              AggExpr("ADD", Term("PAYLOAD", 3, 0), Term("PAYLOAD", 7, 0)), "DENSE", num_groups=50)
    res, exp, tables = run_both(w, fact, host)
    assert res.status() == 0
    compare(w, res, exp)
    one = {d[0]: sjq.build_dim(to_dev(d[1]), d[2], d[3], d[4]) for d in dims}  # one by one: the same tables
    for name, t in tables.items():
        assert t.status() == one[name].status() == 0
        for f, _ in sjq.DimLayout._fields_:
            a, b = getattr(t.layout, f), getattr(one[name].layout, f)
            assert (list(a) == list(b)) if hasattr(a, "__len__") else a == b


def test_launches_of_a_batch_split_by_its_filters_are_all_counted():
    """At most eight dimensions and sixteen filters a launch: 1 + ... + 5, 6 + 7 and 8 filters are three scans and three
    fills; the first tables' builds are one launch for direct tables, one for open addressing."""
    dims = []
    for j in range(8):
        cols = {"k": torch.arange(100, dtype=torch.int32, device="cuda")}
        dims.append((cols, "k", [Pred("k", "GE", 1)] * (j + 1), (),
                     sjq.sjq._BuildOpts(sjq.sjq.FORCE_HASH if j in (1, 7) else 0)))
    tables = sjq.sjq._build_tables(dims)
    assert [sjq.build_launches(t) for t in tables] == [4, 0, 0, 0, 0, 3, 0, 3]
    assert sjq.build_launches(sjq.build_dim(dims[0][0], "k")) == 3
    builder = sjq.TableBuilder(dims[0][0], "k")
    assert sjq.build_launches(sjq.build_tables({"d": builder})["d"]) == 3
    torch.cuda.synchronize()


def test_threads_that_plan_leave_at_most_eight_pieces_of_page_locked_memory_behind():
    """sjq_release counts what it frees: the pieces that finished plans left, whatever thread they ran on."""
    cols, found = to_dev({"k": np.arange(5_000, dtype=np.int32)}), []

    def plan():
        table = sjq.build_dim(cols, "k")
        found.append((table.layout.entries, table.status()))

    def in_threads(n):
        threads = [threading.Thread(target=plan) for _ in range(n)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()

    torch.cuda.synchronize()
    sjq.release()
    for _ in range(3):
        in_threads(1)  # one after the other: the same piece
    assert sjq.release() == 1
    in_threads(16)
    assert 1 <= sjq.release() <= 8
    assert sjq.release() == 0
    plan()
    assert found == [(5_000, 0)] * 20


def test_empty_dimension_in_a_batch():
    empty = {"k": np.zeros(0, np.int32), "p": np.zeros(0, np.int32)}
    full = {"k": np.arange(9, dtype=np.int32), "p": np.arange(9, dtype=np.int32)}
    tables = sjq.sjq._build_tables([(to_dev(d), "k", (), ("p",), sjq.sjq._BuildOpts()) for d in (empty, full, empty)])
    assert [t.layout.entries for t in tables] == [0, 9, 0] and all(t.status() == 0 for t in tables)


@pytest.mark.parametrize("bits,kind", [(2, 9), (4, 8)])
@pytest.mark.parametrize("rows", [0, 1, 5])
def test_a_layout_that_promises_every_key_is_checked_against_any_number_of_rows(bits, kind, rows):
    """Probes of such a table trust the range test alone: keys that are missing would be hits."""
    def promise(L):
        L.kind, L.code_bits, L.npayload = kind, bits, 1
        L.entries, L.kmin, L.kmax, L.slots, L.filter_bits = 6, 0, 5, 6, 128
        L.pay_min[0], L.pay_max[0], L.pay_bits[0] = 0, 2, 2
        L.table_bytes = sjq.layout_bytes(L)

    cols = {"k": np.arange(rows, dtype=np.int32), "p": np.ones(rows, np.int32)}
    assert sjq.build_dim(to_dev(cols), "k", (), ("p",), edit_layout=promise).status() == 21
    cols = {"k": np.arange(6, dtype=np.int32), "p": np.ones(6, np.int32)}
    assert sjq.build_dim(to_dev(cols), "k", (), ("p",), edit_layout=promise).status() == 0


@pytest.mark.parametrize("reuse", [False, True])
def test_builders_alone_and_in_changing_batches(reuse):
    """The same builders in batches of different make-up, alone, and with their columns refreshed on another stream."""
    rng = np.random.default_rng(9)
    n, rows = 20_011, {"a": 4_000, "b": 700, "c": 33_000}
    host = {d: {"k": rng.permutation(r).astype(np.int32), "p": rng.integers(0, 9, r).astype(np.int32),
                "f": rng.integers(0, 9, r).astype(np.int32)} for d, r in rows.items()}
    fact = {d: rng.integers(0, r, n).astype(np.int32) for d, r in rows.items()}
    w = adhoc("batches", fact, [(d, host[d], "k", [Pred("f", "GE", 2)], ["p"]) for d in rows], [(d, d) for d in rows], [],
              KeyExpr((Term("PAYLOAD", 0, 0),)), AggExpr("ADD", Term("PAYLOAD", 1, 0), Term("PAYLOAD", 2, 0)), "DENSE",
              num_groups=9)
    dev = {d: to_dev(c) for d, c in host.items()}
    builders = sjq.workload_builders(w, dev, reuse_layout=reuse)
    refresh = torch.cuda.Stream()
    for turn in range(6):
        for d in rows:  # other payloads in the same range
            host[d]["p"] = rng.permutation(host[d]["p"])
        torch.cuda.synchronize()
        with torch.cuda.stream(refresh):
            for d in rows:
                dev[d]["p"].copy_(torch.from_numpy(host[d]["p"]).pin_memory(), non_blocking=True)
        for b in builders.values():
            b.after(refresh)
        if turn % 3 == 0:
            tables = sjq.build_tables(builders)
        elif turn % 3 == 1:
            tables = sjq.build_tables({d: builders[d] for d in ("c", "a")})
            builders["b"].begin()
            tables["b"] = builders["b"].finish()
            torch.cuda.current_stream().wait_stream(builders["b"].side)
        else:
            tables = {**sjq.build_tables({"b": builders["b"]}), **sjq.build_tables({d: builders[d] for d in ("a", "c")})}
        res, exp, _ = run_both(w, fact, host, tables=tables)
        assert res.status() == 0 and all(t.status() == 0 for t in tables.values())
        compare(w, res, exp)


def test_scratch_of_a_batch_that_grows_is_not_handed_out_while_a_scan_uses_it():
    """With reuse_layout nothing waits for a scan: when a larger batch replaces its lead's scratch, the allocator may not
    give the old block to somebody else before the scans queued on it have run."""
    rng = np.random.default_rng(12)
    dims = {d: to_dev({"k": rng.permutation(n).astype(np.int32), "p": rng.integers(0, 9, n).astype(np.int32)})
            for d, n in (("a", 4_000), ("b", 700), ("c", 900))}
    b = {d: sjq.TableBuilder(c, "k", (), ("p",), reuse_layout=True) for d, c in dims.items()}
    for d in b:
        sjq.build_tables({d: b[d]})
    torch.cuda.synchronize()
    lead, small = b["a"], b["a"].batch_scratch.data_ptr()
    with torch.cuda.stream(lead.scan_side):
        torch.cuda._sleep(400_000_000)  # the scan queued next stays pending for a fifth of a second
    sjq.build_tables({"a": b["a"]})
    tables = sjq.build_tables(b)
    assert lead.batch_scratch.data_ptr() != small
    taken = [torch.empty(sjq.sjq.PLAN_SCRATCH_BYTES, dtype=torch.uint8, device="cuda") for _ in range(64)]
    assert not lead.stats_done[lead.scan].query()  # ... and is pending still
    assert small not in [t.data_ptr() for t in taken]
    torch.cuda.synchronize()
    assert all(t.status() == 0 for t in tables.values())
