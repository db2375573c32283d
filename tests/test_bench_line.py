"""The benchmark's result line is short: a reader that keeps the last 3000 characters of the
output still parses it, whatever the record's other sections hold."""
import json

import bench


def record():
    filler = {f"form_{i}": {"text": "x" * 200, "values": list(range(50))} for i in range(40)}
    return {
        "metric": bench.METRIC, "value": 5.1e11, "unit": bench.METRIC, "n_gpus": 1, "steps": 20,
        "warmup": 5, "ms_per_step": 8.012345678901234, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "tf32x3+f32", "data": "synthetic",
        "config": {"workload": "w" * 120, "form": "lowrank_tf32x3", "l2": "l" * 80,
                   "plan_ms": 22.878080368041992, "parallelism": "replicas x1"},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
        "e2e": {"value": 4.77e11, "unit": bench.METRIC, "h2d_bytes_per_step": 7864320,
                "d2h_bytes_per_step": 163840000},
        "gpu_launches": 2040, "roofline": {"bound": "hbm", "kernel": "lrtc_kernel", "frac": 0.65},
        "cpu_baseline": {"value": 3.4e7, "unit": bench.METRIC, "cores": 16, "kind": "oracle",
                         "sample": "s" * 300},
        "time_to_tol_ms": {"residual_rule": {"tol": 3e-4, "p50": 89.5, "p99": 89.7, "samples": 20,
                                             "iterations": 1070, "percentile_note": "n" * 100},
                           "objective_gap": None, "definition": "d" * 400},
        "reference": {"note": "r" * 300}, "forms": filler, "workloads": filler,
        "err_vs_oracle": {f: {"iterations": 3, "rel_fro": 1.2e-7}
                          for f in ("lowrank_tf32x3", "lowrank_fp32", "dense_bf16x3")},
        "serving": filler, "batching": filler}


def test_line_is_short_and_complete():
    text = json.dumps(bench.result_line(record()))
    assert len(text) < 2000 and "\n" not in text
    line = json.loads(text)
    for key in bench.LINE_KEYS:
        assert key in line
    assert line["e2e"]["h2d_bytes_per_step"] == 7864320 and line["value"] == 5.1e11


def test_line_without_the_optional_sections():
    out = record()
    out["cpu_baseline"] = out["err_vs_oracle"] = None
    out["time_to_tol_ms"]["residual_rule"] = {}
    line = bench.result_line(out)
    assert line["cpu_baseline"] is None and line["err_vs_oracle"] == {}
