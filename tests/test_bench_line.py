"""bench.py's JSON line: one short line with every key of its contract, however
long the record behind it, from a record of the shape a full run makes."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_line_is_short_and_whole():
    forms = {f"form_{i}": {"per_iter_ms_cum": [1.5] * 50, "ms_to_E2": 3.25, "seconds": None} for i in range(12)}
    roof = {"kernel": "k", "bound": "onchip-gather", "achieved": 1.0, "peak": 2.0, "unit": "GB/s", "frac": 0.5,
            "avg_launch_ms": 4.0, "launches_timed": 4, "traffic": None, "def": "x" * 400}
    full = {"metric": bench.METRIC, "value": 600.5, "unit": "GUPS", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 15000.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": bench.workload_config("c5"), "roofline": roof,
            "rooflines": {"project": roof, "backproject": roof}, "cpu_baseline": {"value": 0.01, "sample": "s" * 200},
            "e2e": {"value": 590.0, "unit": "GUPS", "h2d_bytes_per_step": 10, "d2h_bytes_per_step": 5},
            "gpu_launches": 900, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "kernels": {"a": [1.0] * 900}, "measured_onchip": {"fp32_tflops": 77.0, "lds_gbs": 4e4, "how": "h"},
            "secondary": {"config": bench.workload_config("c2"), "value": 650.0, "unit": "GUPS", "ms_per_step": 62.0,
                          "kernels": ["k" * 40] * 90},
            "hbm_kernels": {"x": "y" * 900},
            "time_to_accuracy": {"E2_pmgl_fp32_2iter": 0.0256, "forms": forms,
                                 "literal_rmse_1e-3": {"c1": {"forms": forms}, "c2": {"forms": forms}}},
            "joint_drift_estimation": {"levels": [1.0] * 600}, "oracle_beside": {"o": "p" * 3000}}
    assert len(json.dumps(full)) > 20000
    text = json.dumps(bench.headline(full))
    assert "\n" not in text and len(text) < 6000
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "cpu_baseline"):
        assert line[k] == full[k]
    assert line["roofline"]["frac"] == 0.5 and line["time_to_accuracy"]["ms_to_E2"]["form_3"] == 3.25
    # a run with the optional parts switched off
    for k in ("secondary", "time_to_accuracy", "rooflines", "cpu_baseline", "e2e"):
        full[k] = None
    assert json.loads(json.dumps(bench.headline(full)))["value"] == 600.5
