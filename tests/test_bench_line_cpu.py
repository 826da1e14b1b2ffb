"""The line bench.py prints: every key a reader of it needs, and short whatever tables the record holds."""
import json

import bench
from synthetic import WORKLOADS


def test_headline_is_short():
    table = {f"row{i}": list(range(50)) for i in range(200)}
    row = {"phase": "gram", "kernel": "k", "bound": "hbm", "achieved": 1.0, "peak": 2.0, "unit": "TB/s", "table": table}
    line = {"metric": bench.METRIC, "value": 1.0, "unit": "GB/s", "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 1.0,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": bench.DTYPES["bf16x4"],
            "data": "synthetic", "config": bench.config_dict(WORKLOADS[bench.WORKLOAD], 1e-5, "bf16x4"),
            "gpu_launches": 300000, "gram_tflops": 123.4567, "ranks": [40, 40, 40, 20, 10], "rel_error": 1.2345678901e-06,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 12, "power_w_max": 1234.56},
            "e2e": {"value": 2.0, "unit": "GB/s", "h2d_bytes_per_step": 4, "d2h_bytes_per_step": 5, "raw_h2d": table},
            "methods": {m: {"value": 1.0, "ms_per_step": 2.0, "rooflines": table} for m in ("bf16x4", "fp64")},
            "roofline": row, "rooflines": [row] * 8, "next_rows": table, "configs": table,
            "cpu_baseline": {"value": 1.0, "unit": "GB/s", "cores": 16, "kind": "oracle", "cpu": table}}
    text = json.dumps(bench.headline(line))
    assert len(text) < 1450 and "\n" not in text
    out = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks"):
        assert out[k] == line[k]
    assert out["e2e"] == {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert out["methods"]["fp64"] == {"value": 1.0, "ms_per_step": 2.0}
