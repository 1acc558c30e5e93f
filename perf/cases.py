"""Performance cases of the star-join pipeline: what a user of the library has it do, through its Python binding.

The shapes and sizes are the workload descriptions of datagen.workloads (those of the tests and the benchmark):

  c1  filter + scalar sum, one date join            c4  one join, selectivity x group count sweep
  c2  two filtering joins + date, 7,000 groups      c5  Zipf-skewed int64 keys, open-addressing table
  c3  four joins, 175 groups                        city_pair / city_brand  many possible groups, few survivors

and the ways they are used ("use"):

  run    a repeated query on tables that stand: one fused pass into result buffers that are kept
  step   a repeated query whose dimensions are refreshed: key-range scans, table builds, the fused pass
  adhoc  a query asked once: every table planned and built, result buffers allocated, one fused pass
  list   a hashed group-by whose list is put into key order for what follows on the GPU
  host   fact columns in page-locked host memory, run through in chunks
  merge  the exchange step of a row-sharded query: gathered lists folded into one, in key order

"compiled" asks for the kernel compiled for the query's shape; without it the default options hold (the kernel that
interprets the query's description).  All data are integers, so results are exact.
"""
import itertools
import math
from dataclasses import replace

import torch

import paper_2607_07632_b200 as sjq
from datagen import workloads as W

DEVICE = "cuda:0"
HOST_CHUNK_ROWS = 1 << 22


def listed():
    return [
        # the smallest call: a dashboard tile over one day's rows with default options, all latency
        {"name": "scan_100k", "use": "run", "shape": "c1", "rows": 100_003, "compiled": False},
        # the smallest benchmark configuration
        {"name": "scan_6m", "use": "run", "shape": "c1", "rows": 6_000_000, "compiled": True},
        # an ordinary report: two filtering joins, year x brand
        {"name": "two_join_60m", "use": "run", "shape": "c2", "rows": 60_000_000, "compiled": True},
        # a question asked once, with default options, over a tenth of the largest table
        {"name": "four_join_adhoc_60m", "use": "adhoc", "shape": "c3", "rows": 59_999_999, "compiled": False},
        # the benchmark's step: the largest four-join table, dimensions refreshed every time
        {"name": "four_join_step_600m", "use": "step", "shape": "c3", "rows": 600_000_000, "compiled": True},
        # sweep, middle: one row in ten survives, a group table that fits a block
        {"name": "sweep_10pct_1k_600m", "use": "run", "shape": "c4", "rows": 600_000_000, "below": 1000,
         "groups": 1000, "dim_rows": 3_000_000, "compiled": True},
        # sweep, corner: every row survives into a million groups, returned as an ordered list
        {"name": "sweep_all_1m_600m", "use": "list", "shape": "c4", "rows": 600_000_000, "below": 10000,
         "groups": 1_000_000, "dim_rows": 3_000_000, "compiled": True},
        # 64-bit keys, heavy skew, a table far larger than the caches
        {"name": "skewed_300m", "use": "run", "shape": "c5", "rows": 300_000_000, "dim_rows": 8_000_000,
         "compiled": True},
        # a batch of new rows against a fresh dimension of 8 million sparse keys: the build outweighs the probe
        {"name": "skewed_adhoc_10m", "use": "adhoc", "shape": "c5", "rows": 10_000_019, "dim_rows": 8_000_000,
         "compiled": False},
        # year x city x brand: one row in ten thousand survives, a short ordered list comes back
        {"name": "city_brand_600m", "use": "list", "shape": "city_brand", "rows": 599_999_983, "compiled": True},
        # columns that live in host memory
        {"name": "host_16m", "use": "host", "shape": "c3", "rows": 15_999_989, "compiled": True},
        # eight ranks' lists of a hashed group-by
        {"name": "merge_8x200k", "use": "merge", "shape": "lists", "lists": 8, "groups": 200_000},
    ]


def _spread(rng, lo, hi):
    """A size between lo and hi, evenly over the logarithm; odd sizes as often as not."""
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | rng.randint(0, 1))


def draw(rng):
    use, shape = rng.choice([("run", "c1"), ("run", "c2"), ("run", "c3"), ("run", "c4"), ("run", "c4"), ("run", "c5"),
                             ("run", "city_pair"), ("step", "c2"), ("step", "c3"), ("adhoc", "c3"), ("adhoc", "c5"),
                             ("list", "c4"), ("list", "city_brand"), ("host", "c3"), ("merge", "lists")])
    if use == "merge":
        return {"use": use, "shape": shape, "lists": rng.randint(2, 8), "groups": _spread(rng, 1_000, 200_000)}
    compiled = use != "adhoc" and rng.random() < 0.75
    largest = {"host": 16_000_000}.get(use, {"c1": 60_000_000, "c5": 300_000_000}.get(shape, 600_000_000))
    case = {"use": use, "shape": shape,
            "rows": _spread(rng, 100_000, largest if compiled else min(largest, 60_000_000)), "compiled": compiled}
    if shape == "c4":
        case.update(below=_spread(rng, 1, 10_000),
                    groups=_spread(rng, 10_000, 1_000_000) if use == "list" else _spread(rng, 1, 100_000),
                    dim_rows=_spread(rng, 10_000, 3_000_000))
    if shape == "c5":
        case["dim_rows"] = _spread(rng, 100_000, 8_000_000)
    return case


def _workload(case, seed=W.MASTER_SEED):
    shape, rows = case["shape"], case["rows"]
    if shape == "c4":
        w = W.config4(rows, groups=case["groups"], hashed=case["use"] == "list", dim_rows=case["dim_rows"])
        w = replace(w, preds=(W.Pred("p", "LT", case["below"]),))
    elif shape == "c5":
        w = W.config5(rows, dim_rows=case["dim_rows"])
    else:
        w = {**W.CONFIGS, **W.EXTRA_SHAPES}[shape](rows)
    return replace(w, seed=seed)


def _kept_result(mode, num_groups, capacity, want_count):
    """Result buffers for repeated calls.  A list fills their first entries, as many as there are groups; the rest
    stays zero, so that they can be handed on whole without asking the GPU for the length."""
    res = sjq.alloc_result(mode, num_groups, capacity, want_count, DEVICE)
    if mode == "HASHED":
        for t in (res.keys, res.sums, res.counts):
            t.zero_()
    return res


def prepare(case, seed):
    if case["use"] == "merge":
        n = case["lists"] * case["groups"]
        g = torch.Generator(device=DEVICE).manual_seed(seed)

        def cells(bound):
            return torch.randint(0, bound, (n,), dtype=torch.int64, device=DEVICE, generator=g)

        # groups that most ranks hold, some that few do; spread over the 64-bit keys
        return {"keys": cells(2 * case["groups"]) * 0x9E3779B97F4A7, "sums": cells(1 << 40),
                "counts": cells(1 << 20), "case": case, "result": _kept_result("HASHED", 0, 2 * case["groups"], True)}
    w = _workload(case, seed)
    fact = W.device_fact(w, device=DEVICE)
    dims = {d.name: W.device_dim(w, d, DEVICE) for d in w.dims}
    state = {"case": case, "w": w, "fact": fact, "dims": dims, "opts": sjq.RunOpts(specialise=case["compiled"])}
    if case["use"] == "adhoc":
        return state
    if w.preds:
        state["opts"].pass_ppm = sjq.sample_preds(fact, w.preds)
    if case["use"] == "step":
        state["builders"] = sjq.workload_builders(w, dims, reuse_layout=True)
    else:
        state["tables"] = sjq.build_workload_tables(w, dims)
    if case["use"] == "host":
        state["fact"] = {}
        for name, column in fact.items():
            state["fact"][name] = torch.empty(column.shape, dtype=column.dtype, pin_memory=True).copy_(column)
        state["staging"] = torch.empty(sjq.staging_bytes(state["fact"], HOST_CHUNK_ROWS), dtype=torch.uint8,
                                       device=DEVICE)
    state["result"] = _kept_result(w.mode, w.num_groups, w.capacity, w.agg.want_count)
    return state


def _ordered(res):
    res.sort()
    return {"keys": res.keys, "sums": res.sums, "counts": res.counts, "n": res.n_groups, "status": res.status_dev}


def run(state):
    case = state["case"]
    use = case["use"]
    if use == "merge":
        return _ordered(sjq.merge_groups(state["keys"], state["sums"], state["counts"], 2 * case["groups"],
                                         result=state["result"]))
    w = state["w"]
    if use == "host":
        state["result"], state["host"] = sjq.run_workload_host(
            w, state["fact"], state["tables"], state["staging"], HOST_CHUNK_ROWS, state["opts"],
            result=state["result"], host=state.get("host"))
        torch.cuda.current_stream().synchronize()  # the host copies are read next
        return {"sums": state["host"].sums, "counts": state["host"].counts, "status": state["host"].status}
    if use == "step":
        tables = sjq.build_tables(state["builders"])
    elif use == "adhoc":
        tables = sjq.build_workload_tables(w, state["dims"])
    else:
        tables = state["tables"]
    res = sjq.run_workload(w, state["fact"], tables, state["opts"], result=state.get("result"))
    if use == "list":
        return _ordered(res)
    out = {"sums": res.sums, "counts": res.counts, "status": res.status_dev}
    if use in ("step", "adhoc"):
        out["table_status"] = [t.status_dev for t in tables.values()]
    return out


# share of the rows that each filter of a shape passes on its own, by the fact column it reads
_PASS = {
    "c1": {"orderdate": 365 / 2556, "discount": 3 / 11, "quantity": 29 / 50},
    "c2": {"partkey": 1 / 25, "suppkey": 1 / 5, "orderdate": 1.0},
    "c3": {"custkey": 1 / 5, "suppkey": 1 / 5, "partkey": 2 / 5, "orderdate": 730 / 2556},
    "c4": {"p": 1.0, "fk": 1.0},
    "c5": {"fk": 1 / 4},
    "city_pair": {"custkey": 1 / 25, "suppkey": 1 / 25, "orderdate": 1.0},
    "city_brand": {"custkey": 1 / 5, "suppkey": 1 / 25, "partkey": 1 / 25, "orderdate": 730 / 2556},
}


def work(case):
    """Bytes a pass cannot do without: the first column whole, of a later one the 32-byte sectors that hold a row
    still alive, in the order of filters that reads least; the dimensions where they are built; the result."""
    if case["use"] == "merge":
        return {"bytes": 24 * (case["lists"] + 2) * case["groups"], "flops": 0}
    w = _workload(case)
    passes = dict(_PASS[case["shape"]])
    if case["shape"] == "c4":
        passes["p"] = case["below"] / 10_000
    width = {c.name: 8 if c.is64 else 4 for c in w.fact_cols}
    # (a column filtered on is read once, whether or not its value is used again)
    least = math.inf
    for order in itertools.permutations(passes):
        reach, total = 1.0, 0.0
        for name in order + tuple(c.name for c in w.fact_cols if c.name not in passes):
            total += width[name] * (1.0 - (1.0 - reach) ** (32 // width[name]))
            reach *= passes.get(name, 1.0)
        least = min(least, total)
    size = w.n_rows * least
    for d in w.dims:
        if case["use"] in ("step", "adhoc"):
            used = {d.key, *d.payloads, *(p.col for p in d.preds)}
            size += d.rows * sum(8 if c.is64 else 4 for c in d.cols if c.name in used)
    groups = {"SCALAR": 1, "DENSE": w.num_groups, "HASHED": min(w.num_groups, w.capacity)}[w.mode]
    return {"bytes": size + groups * (24 if w.mode == "HASHED" else 16), "flops": 0}


def tolerance(case):
    return "exact"
