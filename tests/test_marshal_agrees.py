"""The two marshallings of a run's arguments agree: sjq_run gets its structures from the extension module, the other
calls get theirs through ctypes.  In a process of its own a stand-in for sjq_run prints what it is handed, once by the
module and once through ctypes; every option must be set to something else than its default, so that one that is added to
one side only shows here."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STAND_IN = r"""
#include <cstdio>
#include "sjq.h"
typedef long long L;
static void term(const sjq_term &t) { std::printf(" (%d %d %d %lld)", t.src, t.a, t.b, (L)t.mult); }
extern "C" sjq_status sjq_table_info(const sjq_table *, sjq_dim_layout *) { return SJQ_ERR_INVALID_ARG; }
extern "C" sjq_status sjq_run(const sjq_col *fact, int nfact, const sjq_pred *preds, int npreds, const sjq_join *joins,
                              int njoins, const sjq_key_expr *key, const sjq_agg_expr *agg, const sjq_result_spec *spec,
                              const sjq_result *out, const sjq_run_opts *o, void *stream, sjq_run_info *info)
{
    for (int i = 0; i < nfact; ++i) std::printf("col %p %d %lld\n", fact[i].data, fact[i].dtype, (L)fact[i].n);
    for (int i = 0; i < npreds; ++i) {
        std::printf("pred %d %d %lld %lld:", preds[i].col, preds[i].op, (L)preds[i].lo, (L)preds[i].hi);
        for (int k = 0; k < preds[i].nset; ++k) std::printf(" %lld", (L)preds[i].set[k]);
        std::printf("\n");
    }
    for (int i = 0; i < njoins; ++i) std::printf("join %d %p\n", joins[i].fk_col, (const void *)joins[i].table);
    if (key) {
        std::printf("key %d %lld %lld:", key->nterms, (L)key->offset, (L)key->modulo);
        for (int i = 0; i < key->nterms; ++i) term(key->t[i]);
        std::printf("\n");
    }
    std::printf("agg %d %d:", agg->op, agg->want_count);
    term(agg->x), term(agg->y);
    std::printf("\nspec %d %lld %lld\n", spec->mode, (L)spec->num_groups, (L)spec->capacity);
    std::printf("out %p %p %p %p %p %p %zu\n", (void *)out->sums, (void *)out->counts, (void *)out->keys,
                (void *)out->n_groups, (void *)out->status, out->workspace, out->workspace_bytes);
    std::printf("opts");
    sjq_run_opts z = *o; // with the padding at the end cleared
    const unsigned char *b = reinterpret_cast<const unsigned char *>(&z);
    for (size_t i = 0; i < offsetof(sjq_run_opts, l0_bulk) + 4; ++i) std::printf(" %02x", b[i]);
    std::printf("\nstream %p info %d\nend\n", stream, info != nullptr);
    std::fflush(stdout);
    return SJQ_OK;
}
"""

CHILD = r"""
import ctypes, dataclasses, sys
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
from types import SimpleNamespace
import torch
from datagen.workloads import AggExpr, KeyExpr, Pred, Term
import paper_2607_07632_b200.sjq as B
from test_marshal import FakeColumn

stand_in = ctypes.CDLL(sys.argv[2]).sjq_run
fact = {"a": FakeColumn(9, torch.int32, 0x1000), "b": FakeColumn(9, torch.int64, 0x2000)}
event = lambda at: SimpleNamespace(cuda_event=at)
full = B.RunOpts(block_threads=256, ctas_per_sm=3, eager_loads=True, agg_path=2, smem_tables=4096, compaction=2,
                 accumulate=True, order=[2, 0, 1], events=(event(0x71), event(0x72)), specialise=True, rows_per_lane=8,
                 no_filter_bitmap=True, host_copy_all=True, dense_slots=4, group_hash_always=True, warp_agg=1,
                 unfused_scratch=FakeColumn(77, address=0x5000), pass_ppm=(5, 250_000.0, 1_000_000), hot_keys=1,
                 hot_scratch=FakeColumn(99, address=0x6000), l0_bulk=3)
for f in dataclasses.fields(B.RunOpts):
    assert getattr(full, f.name) != getattr(B.RunOpts(), f.name), f.name
queries = [
    dict(preds=(), joins=(), key=None, agg=AggExpr("COL", Term("FACT", "b"), want_count=False), mode="SCALAR", num_groups=1,
         capacity=0),
    dict(preds=[Pred("b", "IN", values=(3, -2**63, 2**63 - 1)), Pred("a", "BETWEEN", -7, 2**40)],
         joins=[("b", SimpleNamespace(handle=0x9000)), ("a", SimpleNamespace(handle=0xa000))],
         key=KeyExpr((Term("PAYLOAD", 1, 1, -25), Term("FACT", "a", 0, 2**62)), offset=-2**62, modulo=97),
         agg=AggExpr("SUB", Term("PAYLOAD", 0, 1, 3), Term("FACT", "a", 0, -1), want_count=True), mode="HASHED",
         num_groups=0, capacity=1234),
]
for q in queries:
    for opts in (None, B.RunOpts(), full):
        hashed = q["mode"] == "HASHED"
        column = lambda at: FakeColumn(5, torch.int64, at)
        res = B.Result(q["mode"], column(0xb0), column(0xc0) if hashed else None, column(0xd0) if hashed else None,
                       column(0xe0) if hashed else None, column(0xf0), FakeColumn(321, address=0x100) if hashed else None)
        assert B.marshal().run(fact, q["preds"], q["joins"], q["key"], q["agg"], B.MODES[q["mode"]], q["num_groups"],
                               q["capacity"], opts, res, 0x42, lambda: None) == 0
        names = list(fact)
        cols = (B._Col * 2)(*[B._Col(t.data_ptr(), int(t.dtype == torch.int64), t.numel()) for t in fact.values()])
        parr, jarr, key, agg, keep = B._query(names, q["preds"], q["joins"], q["key"], q["agg"])
        spec, out = B._ResultSpec(B.MODES[q["mode"]], q["num_groups"], q["capacity"]), B._result_struct(res)
        copts = (opts or B.RunOpts()).to_c()
        ref = ctypes.byref
        assert stand_in(cols, 2, parr, len(q["preds"]), jarr, len(q["joins"]), ref(key) if key is not None else None, ref(agg),
                        ref(spec), ref(out), ref(copts), ctypes.c_void_p(0x42), ref(res.info)) == 0
"""


def test_the_extension_module_and_ctypes_pass_the_same_arguments(tmp_path):
    from paper_2607_07632_b200 import build

    build.build()
    (tmp_path / "stand_in.cpp").write_text("#include <cstddef>\n" + STAND_IN)
    (tmp_path / "child.py").write_text(CHILD)
    lib = str(tmp_path / "libstand_in.so")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I" + os.path.join(ROOT, "include"),
                           str(tmp_path / "stand_in.cpp"), "-o", lib])
    run = subprocess.run([sys.executable, str(tmp_path / "child.py"), ROOT, lib], capture_output=True, text=True, timeout=300,
                         env={**os.environ, "LD_PRELOAD": lib}, cwd=ROOT)
    assert run.returncode == 0, run.stderr[-3000:]
    calls = run.stdout.split("end\n")[:-1]
    assert len(calls) == 12
    for module, through_ctypes in zip(calls[::2], calls[1::2]):
        assert module == through_ctypes
    assert len(set(calls)) == 4  # two queries, no options or the default ones, and all of them
