"""The line that bench.py prints on standard output has to fit a reader that keeps its last 3,000 characters."""
import json

import bench


def _line():
    plan = {"order": [12] * 9, "in_smem": [1] * 9, "first_sparse_stage": 1, "queue_levels": 3, "agg_path": "shared",
            "grid": 148, "block": 1024, "smem_bytes": 231_424, "kernel_launches": 12}
    f = 472641622758.3547
    return {"metric": bench.METRIC, "value": f, "unit": bench.UNIT, "n_gpus": 8, "steps": 200, "warmup": 10,
            "ms_per_step": 1.2694607734680177, "higher_is_better": True, "scaling": "strong", "vs_baseline": None,
            "dtype": "int64", "data": "synthetic",
            "config": {"workload": "c4_sweep_s0.0001_g1000000_hashed", "rows_per_gpu": 1_200_000_000, "rows_total": 9_600_000_000,
                       "referenced_bytes_per_row": 24,
                       "step": "scan + build of every dimension table, then the fused pass, then all-gather of the "
                               "per-rank group lists and a merge kernel",
                       "l2": "inputs (14.4 GB) exceed the 126 MB L2; no flush needed",
                       "parallelism": "row-sharded x8, dimensions replicated", "plan": plan,
                       "fused_kernel": "compiled for the query during warm-up"},
            "effective_gbs": f, "pct_of_8tbs": f, "pct_of_measured_copy_peak": f, "parity": True,
            "roofline": {"bound": "hbm", "kernel": "sjq_jit_kernel", "achieved": f, "peak": f, "peak_kind": "of measured",
                         "unit": "GB/s", "frac": 0.7246661436767854, "traffic": f,
                         "traffic_source": "the plan that ran differs from the one captured in profiles/fused_kernel_c3_100m.md",
                         "algorithmic_bytes_per_row": f, "kernel_ms": f, "bytes_per_row_64B_model": f,
                         "note": "achieved, frac: 32-byte-sector model",
                         "pass_fractions": {str(i): 0.123456 for i in range(6)}, "effective_gbs_kernel": f},
            "cpu_baseline": {"value": f, "unit": bench.UNIT, "cores": 1, "kind": "oracle",
                             "sample": "first 100000000 fact rows of the workload; row loop 60.40 s + dimension maps 10.15 s",
                             "host_cores_available": 128},
            "e2e": {"value": f, "unit": bench.UNIT, "h2d_bytes_per_step": 17_580_925_535, "h2d_copied_bytes": 17_200_000_000,
                    "h2d_dimension_bytes": 1_200_000_000, "h2d_in_place_bytes_estimate": 1_380_925_535,
                    "columns": {c: "not transferred" for c in ("custkey", "suppkey", "partkey", "orderdate", "revenue", "supplycost")},
                    "d2h_bytes_per_step": 12_804, "ms_per_step": f, "steps": 3, "chunk_rows": 33_554_432,
                    "matches_device_run": True,
                    "api": "sjq_run_host: pinned columns in chunks, sparse ones read in place, result copied back"},
            "gpu_launches": 123_456, "clocks": {"sm_mhz": 1965, "sm_max_mhz": 1965, "reasons": ["sw_power_cap", "gpu_idle"], "samples": 300}}


def test_the_line_is_short_and_whole_and_the_points_go_to_standard_error(capsys):
    points = [{"workload": f"c4_sweep_s0.0001_g{i}_hashed", "parity": i != 3, "ms_min": 1.23456789012} for i in range(27)]
    bench.print_line(_line(), points, [{"variant": "v" * 5000}])
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 2900
    line = json.loads(out)
    assert set(_line()) | {"points"} == set(line) and abs(line["value"] / 472641622758.3547 - 1) < 1e-6
    assert line["points"] == {"run": 27, "parity": 26, "without_parity": ["c4_sweep_s0.0001_g3_hashed"]}
    rows = [json.loads(r) for r in err.splitlines()]
    assert [list(r) for r in rows] == [["point"]] * 27 + [["ablation"]] and rows[5]["point"]["workload"].endswith("g5_hashed")
