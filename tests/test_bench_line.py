"""The benchmark's last output line: every required key, and short enough to be
read whole where only the last 2000 characters of an output are kept."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_headline_is_short_and_complete():
    f = 123456789012.34567
    shape = {"shape": [11, 8, 128, 8], "ctas": 152, "threads": 640, "ms_per_step": 0.1234567890123456}
    line = {
        "metric": bench.METRIC, "value": f, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5,
        "ms_per_step": 46.123456789012345, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic (seeded obstacles)",
        "config": {"workload": bench.WORKLOAD, "grid": [128, 128, 64, 96], "horizon_s": 2.0, "cfl": 0.8,
                   "time_steps_per_solve": 352, "step": "x" * 75, "l2": "y" * 75, "parallelism": "replicas x8",
                   "tile": {**shape, "tried": [shape] * 34}},
        "roofline": {"bound": "hbm", "achieved": f, "peak": f, "unit": "GB/s", "frac": 0.9012345678901234,
                     "traffic": {"bytes": f, "source": "z" * 120}, "kernel": "hj_step_tiled_kernel",
                     "peak_source": "measured hbm_gbs", "bytes_per_update": 8, "avg_launch_ms": 0.1312345678901234},
        "latency_ms": {"p50": 46.12345678901234, "p99": 46.12345678901234},
        "accuracy": {"big": [f] * 300},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 100,
                   "power_w_max": 1057.1},
        "gpu_launches": 7120,
        "e2e": {"value": f, "unit": bench.UNIT, "h2d_bytes_per_step": 805306368, "d2h_bytes_per_step": 805306368,
                "ms_per_step": 54.12345678901234},
        "serving": {"sweep": [{"rate": f, "p99": f}] * 200},
    }
    text = json.dumps(bench.headline(line), default=bench.json_default)
    assert len(text) < 1990
    out = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert out[key] == line[key] or key == "config"
    assert "tried" not in out["config"]["tile"] and line["config"]["tile"]["tried"]  # the detail line keeps it
