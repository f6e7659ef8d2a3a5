"""The line that bench.py prints is short enough for a caller that keeps the last
1,500 characters of the output, whatever the complete record holds (CPU)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_headline_is_short_and_complete():
    long = 0.12345678901234567
    config = {"workload": "sinusoid_8d_N1000000_n50", "N": 1000000, "p": 8, "M": 100000, "n0": 6,
              "n": 50, "N_close": 1000, "theta": 1.0, "g": 1e-06, "search": "ray", "nrays": 8,
              "precision": "fp32 scoring, fp64 update",
              "l2": "flushed: 256 MB written before every step",
              "parallelism": "locations sharded over 1 rank(s)"}
    record = {"metric": "locations/sec at N=1e6,d=8,n=50 (ray search)", "value": 1e5 + long,
              "unit": "locations/s", "n_gpus": 1, "steps": 20, "warmup": 5,
              "ms_per_step": 149 + long, "higher_is_better": True, "scaling": "weak",
              "vs_baseline": None, "dtype": "f32/f64",
              "data": "synthetic (seeded uniform design, sinusoid-plus-product response)",
              "config": config, "rmse": long, "gpu_launches": 240,
              "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 20},
              "e2e": {"value": 6e5 + long, "unit": "locations/s", "h2d_bytes_per_step": 78400000,
                      "d2h_bytes_per_step": 1600000},
              "roofline": {"kernel": "ray32", "bound": "alu", "achieved": 15 + long,
                           "peak": 80.54784, "unit": "TFLOP/s", "frac": long, "traffic": None,
                           "peak_source": "x" * 60, "flop_count": "x" * 80, "launch_ms": long},
              "cpu_baseline": {"value": 130 + long, "unit": "locations/s", "cores": 16,
                               "kind": "oracle", "sample": "x" * 60, "one_core": {}},
              "kernels": {"k%d" % i: {"ms_per_step": long, "launches": 5, "share": long}
                          for i in range(12)},
              "other_forms": {"f%d" % i: {"text": "x" * 900} for i in range(9)},
              "serving_form": {"rates": [{"text": "x" * 300}] * 15}}
    line = bench.headline(record)
    assert len(json.dumps(record)) > 10_000 and len(json.dumps(line)) < 1500
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
                "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
                "gpu_launches", "clocks"):
        assert line[key] == record[key]
    assert line["roofline"]["frac"] == long and line["cpu_baseline"]["kind"] == "oracle"
