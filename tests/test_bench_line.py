"""The line that bench.py prints is one JSON object with the keys its readers
look for, and short: they keep only the last few thousand characters."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

X = 1234567890.1234567


def record(bench):
    text = "x" * 200
    oracle = {"value": X, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": text}
    return {
        "metric": bench.METRIC, "value": X, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": X,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": dict(bench.headline_config(8), l2=text[:80]), "gp_stages_per_s": X,
        "error_vs_oracle": {"psi_rel_l2": X, "q_abs": X, "p_abs": X, "sample": text[:100]},
        "roofline": {"bound": "alu", "achieved": X, "peak": X, "unit": "TFLOP/s", "frac": X, "traffic": X, "kernel": text[:80],
                     "flops_per_point_stage": X, "note": text, "peak_source": text, "fp32_fma_tflops_measured": X,
                     "hbm": {"achieved": X, "peak": X, "unit": "GB/s", "frac": X, "peak_source": text,
                             "bytes_per_point_stage": 64}},
        "cpu_baseline": dict(oracle, all_cores=dict(oracle, sample=text[:120])),
        "e2e": {"value": X, "unit": bench.UNIT, "h2d_bytes_per_step": 6879707136, "d2h_bytes_per_step": 6879707136,
                "note": text},
        "gpu_launches": 20, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 300},
        "wall_s": X,
    }


def test_the_line_is_short_and_complete():
    import bench

    text = bench.contract_line(record(bench))
    assert "\n" not in text and len(text) < bench.LINE_LIMIT
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks"):
        assert key in line
    assert line["e2e"]["h2d_bytes_per_step"] > 0 and "frac" in line["roofline"]["hbm"]
