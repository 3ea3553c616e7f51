"""The benchmark's printed line: every key of the contract, and short enough
to survive in the tail of a log."""
import json

import bench


def test_short_line():
    full = {k: 1.0 for k in bench.CONTRACT}
    full["config"] = {"workload": bench.workload_desc("assembly1m"), "mode": "mixed", "parallelism": "single",
                      "l2": "256 MB flush between timed steps"}
    full["stage_ms"] = {k: 123.456789012345 for k in "abcdef"}
    full["clocks"] = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 12}
    full["e2e"] = {"value": 302.0123456789, "unit": "ms", "h2d_bytes_per_step": 32000640,
                   "d2h_bytes_per_step": 2863789032, "runs": 5, "stage_ms_last": {"ms_total": 1.0}}
    full["roofline"] = {"bound": "alu", "kernel": "k_accum_f32", "achieved": 11.5, "peak": 80.5, "unit": "TFLOP/s",
                        "frac": 0.14, "ms_per_launch": 26.0, "peak_source": "x" * 200}
    full["batch_form"] = {"ms_per_batch": 1.0, "workload": "x" * 500}
    full["readings_form"] = {"rows": [{"x": 1.0}] * 1000}
    full["autotune"] = "y" * 5000
    full["adaptive_form"] = None   # not measured
    line = json.loads(json.dumps(bench.short_line(full)))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert k in line
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
    assert {"sm_mhz", "sm_max_mhz", "reasons"} <= set(line["clocks"])
    assert "readings_form" not in line and "adaptive_form" not in line
    assert len(json.dumps(line)) < 2500
