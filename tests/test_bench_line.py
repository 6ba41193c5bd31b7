"""bench.py prints one line that a reader of the output's end gets whole, with
every key of the contract."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_the_printed_line_is_short_and_complete():
    x = 12345.678901234567
    note = "n" * 400
    line = {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5,
            "ms_per_step": x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "dtype_note": note, "data": "synthetic", "config": bench.config(8), "latency_ms": {"p50": x, "p99": x},
            "split_ms": {"setup": x, "solve": x}, "levels": {"n": list(range(64))}, "lambda2": x / 1e9, "residual": x,
            "roofline": {"bound": "alu", "kernel": "k_power_sell<double, int>, level-0 launch", "achieved": x,
                         "peak": x, "unit": "TFLOP/s", "frac": x, "traffic": 794075392, "note": note},
            "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 1, "kind": "oracle", "sample": note},
            "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 79280008, "d2h_bytes_per_step": 8000000,
                    "host_memory": "pinned"},
            "gpu_launches": 123456, "host": {"model": note},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 99},
            "fp32": {"value": x, "dtype": note}, "accuracy_vs_oracle": {"c2_fp64": {"vec_rel_err": x / 1e19}},
            "c1": {"value": x}, "batch": {"fp32": {"value": x}}, "serving": {"fp32": {"saturation_solves_s": x}},
            "chung_lu": {"fp32": {"value": x}}, "gcmg": [note], "schedule_study": [note] * 40}
    out = bench.headline(line)
    text = json.dumps(out)
    assert len(text) < 2000
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert key in out
    assert out["config"] == bench.config(8)
    assert abs(out["value"] - x) <= 1e-5 * x
    assert set(out["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert set(out["clocks"]) == {"sm_mhz", "sm_max_mhz", "reasons"}
    none = dict(line, e2e=None, cpu_baseline=None, fp32=None, accuracy_vs_oracle=None, c1=None, batch=None,
                serving=None, chung_lu=None)
    assert bench.headline(none)["others"]["fp32"] is None
