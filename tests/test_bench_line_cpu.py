"""The bench's one line stays short however long its tables are."""
import json

import bench

KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
        "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "kernel_share", "launch")


def test_summary_line_drops_the_tables_only():
    table = {str(k): {"max_abs": 1e-6 * k, "sign_agreement": 1.0} for k in range(300)}
    out = {k: k for k in KEYS}
    out["config"] = {"workload": "w" * 200}
    out["fp64_path"] = {"value": 393.0, "marginal_error_per_layer": {"layers": table, "max_abs": 6e-6}, "note": "n" * 200}
    out["batched"] = {"16x_n1000": {"instance_layers_per_s": 2600.0, "errors": table, "list": list(range(1000))}}
    out["scale"] = None
    line = bench.summary_line(out)
    assert all(line[k] == out[k] for k in KEYS)
    assert line["fp64_path"] == {"value": 393.0, "marginal_error_per_layer": {"max_abs": 6e-6}}
    assert line["batched"] == {"16x_n1000": {"instance_layers_per_s": 2600.0}}
    assert line["scale"] is None
    assert len(json.dumps(out)) > 20000 and len(json.dumps(line)) < 2000
