"""The benchmark's result line: one short line of strict JSON whatever the
size of the record behind it."""
import json
import math

import bench


def test_result_line_is_short_and_strict():
    record = {
        "metric": bench.METRIC, "value": 2.5e10, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 12.5, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": "w" * 300, "l2": "flushed", "seed": 1234},
        "chosen_fp32": {"value": 1e11, "unit": bench.UNIT, "ms_per_step": 1.0, "dtype": "f32", "clocks": {"sm_mhz": 1},
                        "compiled_shape_by_p": {str(p): p for p in range(18)}},
        "time_to_rel_1e-4_s": {"p": 10, "plain_fp64": math.nan, "chosen_fp32": 0.1, "method": "m" * 300},
        "error_vs_ed_per_p_s": {"by_p": {p: [{"amp": math.inf}] * 100 for p in range(18)}},
        "roofline": {"bound": "alu", "achieved": 30.0, "peak": 75.0, "unit": "TFLOP/s", "frac": 0.4, "kernel": "k", "note": "n" * 2000},
        "cpu_baseline": {"value": 6e7, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "per_config": {"x": ["y" * 5000]}},
        "e2e": {"value": 2.4e10, "unit": bench.UNIT, "h2d_bytes_per_step": 8000, "d2h_bytes_per_step": 32004}, "gpu_launches": 40,
        "several_coordinates": {"rows": [1.0] * 5000}, "clocks": {"sm_mhz": 2000, "sm_max_mhz": 2070, "reasons": []},
    }
    text = bench.result_line(record)
    assert "\n" not in text and len(text) < 2500
    line = json.loads(text, parse_constant=lambda c: 1 / 0)   # no NaN, no Infinity
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert k in line
    assert line["value"] == 2.5e10 and line["e2e"] == record["e2e"] and line["time_to_rel_1e-4_s"]["plain_fp64"] is None
