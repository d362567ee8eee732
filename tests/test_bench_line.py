"""The line that the benchmark prints on standard output: every key of its contract, short enough to be
read from the end of the output, whatever the extras' tables hold."""
import json

import bench


def test_headline_is_short_and_complete():
    table = {f"kernel_{k}": {f"field_{j}": 1.0 / (3 + j + k) for j in range(30)} for k in range(20)}
    line = {
        "metric": bench.METRIC, "value": 33.123456789012345, "unit": "solves/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 30.123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32 inner, f64 outer", "data": "synthetic",
        "config": {"workload": bench.WORKLOAD_C2, "method": "m" * 200, "grid": [512, 512, 512], "tol": 1e-8,
                   "inner_tol": 4e-5, "density_ratio": 7.6, "l2": "inputs larger than L2 (~15.4 GB working set)",
                   "replicas": 1},
        "gpu_launches": 2400, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"]},
        "roofline": {"bound": "hbm", "achieved": 1 / 3, "peak": 6793.1, "unit": "GB/s", "frac": 0.93, "traffic": 3.6e9,
                     "kernel": "k" * 40, "timing": "t" * 400},
        "e2e": {"value": 26.27, "unit": "solves/s", "h2d_bytes_per_step": 1 << 30, "d2h_bytes_per_step": 1 << 30},
        "cpu_baseline": {"value": 1 / 7, "unit": "solves/s", "kind": "oracle", "sample": "s" * 300},
        "iterations": 12, "outer_iterations": 3, "rel_res": 1 / 3, "solve_ms_median": 1 / 3, "solve_hbm_frac": 1 / 3,
        "kernels": table, "c1_256": table, "serving": {"error": "RuntimeError: " + "x" * 500}, "batch": table,
        "summary": {f"figure_{k}": 1.0 / (3 + k) for k in range(14)},
    }
    short = bench.headline(line)
    text = json.dumps(short)
    assert len(text) < 2600  # readers were seen to keep the last 3000 characters
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline"):
        assert key in short
    assert short["value"] == line["value"] and short["ms_per_step"] == line["ms_per_step"]
    assert short["config"] == line["config"] and short["e2e"] == line["e2e"]
    assert short["failed"] == ["serving"] and "kernels" not in short
