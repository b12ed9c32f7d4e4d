"""The line bench.py prints: short enough to be read whole from the end of a log, with every key of its contract."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_headline_is_short_and_complete():
    long = {f"detail_{i}": [0.123456789012345] * 20 for i in range(20)}
    figures = {"bound": "hbm", "achieved": 1234.56789012, "peak": 6781.8, "unit": "GB/s", "frac": 0.5, "kernel": "phase_a"}
    record = {"metric": bench.METRIC, "metric_detail": bench.METRIC_DETAIL, "value": 4024.0672294939022, "unit": "GB/s",
              "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 2.134639930725098, "higher_is_better": True,
              "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
              "config": {"workload": "512x512x512", "shape": [512] * 3, "parallelism": "single GPU"},
              "roofline": {**figures, **long}, "cpu_baseline": {"value": 3.15, "unit": "GB/s", **long},
              "e2e": {"value": 1246.624107361177, "unit": "GB/s", "h2d_bytes_per_step": 1 << 30, "d2h_bytes_per_step": 1 << 30},
              "gpu_launches": 80, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
              "serving": {"p50_ms": 1.346047, "p99_ms": 15.81079424, **long},
              "secondary": {name: {"value": 1000.0 / 3, "ms_per_step": 7.0 / 3, "roofline": figures, **long}
                            for name, _, _ in bench.SECONDARY}}
    line = bench.headline(record)
    assert len(json.dumps(line)) < 4000 < len(json.dumps(record))
    for key in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                "config", "e2e", "gpu_launches", "clocks", "value", "ms_per_step"):
        assert line[key] == record[key], key
    assert line["roofline"]["frac"] == 0.5 and line["serving"] == {"p50_ms": 1.34605, "p99_ms": 15.8108}
    assert set(line["secondary"]) == set(record["secondary"])
