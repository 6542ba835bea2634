"""The line that bench.py prints for its own arm: the contract's keys, and short
whatever was measured beside them."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_line_keeps_the_contract_and_stays_short(tmp_path):
    wl, k, K = bench._workload("medium", 0)
    x = 1234567890.123456789
    detail = {f"key_{i}": {"value": x, "note": "n" * 80} for i in range(60)}
    comp = {"ms_per_step": x, "tnn_speedup": x, "identical_neighbours": True, "alu": detail}
    out = {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 1, "steps": 400, "warmup": 5,
           "ms_per_step": x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
           "data": "synthetic",
           "config": dict(bench._config(wl, k, K, "medium"),
                          tuning={"seed_segments": 4, "seed_window": 0, "extra": 4, "sweep": False, "defer_cells": x},
                          parallelism="replicas x1: each rank its own window"),
           "clocks": {"sm_mhz": x, "sm_max_mhz": x, "reasons": ["sw_power_cap"], "samples": 100},
           "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 6400000, "d2h_bytes_per_step": 102400000,
                   "ms_per_step": x, "includes": "i" * 300},
           "gpu_launches": 1200,
           "roofline": dict(detail, bound="alu", achieved=x, peak=x, unit="T FP32 lane-ops/s", frac=x, traffic=None,
                            kernel="k_tnn_grid_search", kernel_ms=x),
           "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "cpu": "c" * 40,
                            "sample": "s" * 200, "parity": dict(detail, queries_checked=8192, identical_indices=True)},
           "comparator": {"tensor_core": comp, "cuda_core": comp}, "stats_per_step": detail, "e2e_breakdown": detail,
           "tc_tiles": detail, "nowcast": detail, "precision": detail}
    line = bench._line(out)
    text = json.dumps(line)
    assert len(text) < 2500
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches"):
        assert line[key] == out[key]
    for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == out["e2e"][key]
    path = tmp_path / "sub" / "details.json"
    bench._write_details(out, str(path))
    assert json.loads(path.read_text()) == out


def test_line_without_the_optional_measurements():
    out = {"metric": bench.METRIC, "value": 1.0, "unit": bench.UNIT, "n_gpus": 2, "steps": 3, "warmup": 3,
           "ms_per_step": 1.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
           "data": "synthetic", "config": {}, "clocks": None, "e2e": {"value": 1.0, "unit": bench.UNIT},
           "gpu_launches": 9, "roofline": None, "cpu_baseline": None, "comparator": None}
    line = bench._line(out)
    assert line["cpu_baseline"] is None and line["comparator"] == {} and line["n_gpus"] == 2
