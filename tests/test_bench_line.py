"""bench.py's line on stdout stays short, whatever is measured beside the headline."""
from __future__ import annotations

import json


def test_headline_is_short_and_whole():
    import bench
    entry = {"dtype": "f64", "value": 5e3, "unit": "GB/s", "ms_per_step": 70.0, "hbm_frac_of_measured": 0.5, "estimate": -1e6,
             "rel_err_vs_exact": 1e-4, "phase_ms": {}, "roofline": {"kernel": "k" * 500}}
    line = {key: 1.0 for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                                 "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "e2e")}
    line.update(precisions={p: dict(entry) for p in ("df64", "f64", "f32")}, workloads={"c1": ["x" * 40000]})
    line["c3_time_to_1e-3"] = {"ms": [1.0] * 100}
    short, details = bench.split_line(line)
    assert len(json.dumps(short)) < 2000
    assert all(key in short for key in line if key not in ("workloads", "c3_time_to_1e-3"))
    assert set(short["precisions"]) == {"df64", "f64", "f32"} and short["precisions"]["f32"]["ms_per_step"] == 70.0
    assert details["details"]["workloads"] == line["workloads"] and details["details"]["precisions"] == line["precisions"]
