"""bench.py's one line of output: the headline figures and nothing that grows
with the number of sections measured (a line of 27,000 characters was cut by
its reader and lost).  No GPU."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2506_18579_gb300 import workloads as wl  # noqa: E402


def _full(x=123456789.123456789):
    many = {"section %d" % i: {"ms": x, "rays_per_s": x} for i in range(300)}
    return {
        "metric": bench.METRIC, "value": x, "unit": "rays/s", "n_gpus": 8, "steps": 1000, "warmup": 100, "ms_per_step": x,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": wl.config2(elev_step=6.0, az_step=60.0).name, "rays": 24840, "precision": "mixed",
                   "rtol": 1e-8, "launch": {"kernel": 1, "stencil": 3, "block_threads": 128, "order": 1, "lanes_per_ray": 4},
                   "l2": "flushed (512 MiB write) before every timed step", "parallelism": "replicas"},
        "ray_steps_per_s": x, "fan_latency_ms": {"p50": x, "p99": x},
        "e2e": {"value": x, "unit": "rays/s", "h2d_bytes_per_step": 12345678, "d2h_bytes_per_step": 12345678},
        "gpu_launches": 2000, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 99999,
                                         "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_power_cap"]},
        "roofline": {"bound": "alu", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "traffic": 27159040, **many},
        "cpu_baseline": {"value": x, "unit": "rays/s", "cores": 128, "kind": "oracle", "seconds": x, **many},
        "accuracy": {"vs_cpu_oracle": {"rays_compared": 24706, "status_mismatch": 0, "p_and_d_within_bar_share": x, **many},
                     **many}, "batch": many, "serving": many}


def test_headline_is_short_and_whole():
    full = _full()
    line = bench.headline(full)
    text = json.dumps(line)
    assert len(text) <= bench.HEADLINE_CHARS and "\n" not in text
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert k in line
    assert abs(line["value"] / full["value"] - 1) < 1e-6 and line["config"] == full["config"]
    assert set(line["clocks"]) == {"sm_mhz", "sm_max_mhz", "reasons"}
    assert set(line["e2e"]) == set(full["e2e"])
    assert line["accuracy"]["status_mismatch"] == 0
    none = bench.headline({**full, "cpu_baseline": None, "accuracy": {}})  # more than one GPU: no CPU leg
    assert none["cpu_baseline"] is None and "accuracy" not in none
