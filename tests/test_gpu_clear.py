"""A pass that clears its result while its clear is late: the waits of the other blocks run out, which the status tells, and
the words are left as the next run, or the replay of a captured one, needs them."""
import pytest
import torch

pytestmark = pytest.mark.gpu

sjq = pytest.importorskip("paper_2607_07632_b200") if torch.cuda.is_available() else None

from gpuhelpers import compare, oracle_result, to_dev  # noqa: E402
from test_gpu_forms import _grouped, _query  # noqa: E402

ASYNC_WAIT = 22


def _late(ms, **options):
    class Late(sjq.RunOpts):
        def to_c(self):
            o = super().to_c()
            o.sync_late_ms = ms
            return o

    return Late(host_copy_all=True, **options)


# left: what the words hold before the first run
@pytest.mark.parametrize("groups,compiled,left", [(0, False, -1), (0, True, 0), (20, False, 1 << 21), (20, True, -1),
                                                  (3_000, False, 0), (3_000, True, 1 << 21)])
def test_a_clear_that_comes_late_is_told(groups, compiled, left):
    n = 100_003
    fact = _grouped(n, max(1, groups), groups)
    w = _query(fact, groups)
    exp = oracle_result(w, fact, {})[1]
    dev = to_dev(fact)
    options = dict(specialise=compiled, agg_path=1 if groups > 1 else 0)
    res = sjq.run_workload(w, dev, {}, sjq.RunOpts(**options))
    assert res.info.kernel_launches == 1
    host = {c: torch.from_numpy(v).pin_memory() for c, v in fact.items()}
    staging = torch.empty(sjq.staging_bytes(host, 2**17), dtype=torch.uint8, device="cuda")
    words = res.sync = torch.full((8,), left, dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        sjq.run_workload(w, dev, {}, sjq.RunOpts(**options), result=res)

    def through_host(ms):
        for t in (res.sums, res.counts, res.status_dev):
            t.fill_(77)
        sjq.run_workload_host(w, host, {}, staging, 2**17, _late(ms, **options), result=res)
        torch.cuda.synchronize()
        assert words[0] == 0 and ((words == 0) | (words == left)).all()
        return res.status()

    assert through_host(3_000) == ASYNC_WAIT
    for _ in range(2):
        res.sums.fill_(5)
        graph.replay()
        torch.cuda.synchronize()
        assert res.status() == 0
        compare(w, res, exp)
    assert through_host(0) == 0
    compare(w, res, exp)
    assert through_host(20) == 0  # late, and waited for
    compare(w, res, exp)


def test_runs_behind_other_kinds_of_work_in_a_capture():
    """A clear, and a pass that clears, follow a copy, a fill, a kernel and another stream's work."""
    big, small = 2**19 + 5, 10_007
    for n in (small, big):
        fact = _grouped(n, 50, n)
        w, src = _query(fact, 50), to_dev(fact)
        exp = oracle_result(w, fact, {})[1]
        for compiled in (False, True):
            opts = sjq.RunOpts(specialise=compiled, agg_path=1)
            dev = {c: torch.zeros_like(t) for c, t in src.items()}
            res = sjq.run_workload(w, dev, {}, opts)
            other = torch.cuda.Stream()
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph):
                here = torch.cuda.current_stream()
                other.wait_stream(here)
                with torch.cuda.stream(other):
                    dev["p"].copy_(src["p"])
                dev["g"].zero_()
                dev["g"].add_(src["g"])
                dev["m"].copy_(src["m"])
                here.wait_stream(other)
                sjq.run_workload(w, dev, {}, opts, result=res)
                kept = res.sums.clone()
                res.sums.zero_()
                sjq.run_workload(w, dev, {}, opts, result=res)
            for _ in range(3):
                for t in dev.values():
                    t.zero_()
                res.sums.fill_(9)
                graph.replay()
                torch.cuda.synchronize()
                assert res.status() == 0
                compare(w, res, exp)
                assert torch.equal(kept, res.sums)
