"""Work that waits in the SMs for a long pass leaves other streams their room."""
from dataclasses import replace

import pytest
import torch

from datagen import workloads as W

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None


def _query(w):
    fact = W.device_fact(w)
    tables = sjq.build_workload_tables(w, {d.name: W.device_dim(w, d) for d in w.dims})
    opts = sjq.RunOpts(specialise=True, pass_ppm=sjq.sample_preds(fact, w.preds) if w.preds else ())
    res = sjq.alloc_result(w.mode, w.num_groups, w.capacity, w.agg.want_count, "cuda")
    return lambda: sjq.run_workload(w, fact, tables, opts, result=res)


def test_a_large_clear_behind_a_long_pass():
    """The calls of another stream take as long beside a long pass and the clear of eight million groups, in turn, as beside
    long passes alone; eight waiting blocks of the clear per SM made them take more than one and a half times as long."""
    long_pass = _query(W.config1(200_000_000))
    clear = _query(replace(W.config4(100_000, groups=8_000_000, hashed=False, dim_rows=1000), preds=(W.Pred("p", "LT", 100),)))
    other = _query(W.config2(2_000_000))
    side = torch.cuda.Stream()

    def beside(*mains):
        took = []
        for _ in range(4):
            start, a, b = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            torch.cuda.synchronize()
            start.record()
            for _ in range(30):
                for m in mains:
                    m()
            with torch.cuda.stream(side):
                side.wait_event(start)
                a.record()
                for _ in range(60):
                    other()
                b.record()
            torch.cuda.synchronize()
            took.append(a.elapsed_time(b))
        return min(took)

    assert beside(long_pass, clear) < 1.25 * beside(long_pass)
