"""The benchmark's printed line: the contract's keys whole, the other
workloads in short, and short enough to be kept as the tail of a log."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_printed_line():
    import bench
    base = {"metric": "m" * 84, "value": 1331815757611.4624, "unit": "points/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.8062378, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "w" * 600}, "roofline": {"bound": "alu", "frac": 0.8644659},
            "e2e": {"value": 1.2e12, "unit": "points/s", "h2d_bytes_per_step": 50331648, "d2h_bytes_per_step": 4194304},
            "gpu_launches": 20, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}}
    table = {f"v{i}": {"points_per_s": 1.0 / 3, "note": "n" * 100} for i in range(100)}
    one = dict(base, max_norm_err=1e-7, tables=table)
    short = bench.short_line(dict(base, variants=table, configs={k: one for k in ("plain", "batch", "tensor", "fit")}))
    for k, v in base.items():
        assert short[k] == bench._rounded(v)
    assert abs(short["value"] / base["value"] - 1) < 1e-6 and isinstance(short["n_gpus"], int)
    assert "variants" not in short and set(short["configs"]) == {"plain", "batch", "tensor", "fit"}
    assert short["configs"]["fit"]["frac"] == base["roofline"]["frac"] and "tables" not in short["configs"]["fit"]
    assert len(json.dumps(short)) < 2800
    run = bench.short_line({k: base[k] for k in base if k != "e2e"})
    assert "e2e" not in run and "configs" not in run
