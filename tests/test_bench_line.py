"""The line that bench.py prints on stdout: every key of the contract, and short
enough that the last 2,500 characters of the output hold it, however much is
measured beside it."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline")


def test_the_line_keeps_the_contract_and_is_short():
    sys.path.insert(0, ROOT)
    import bench
    line = {k: 1.0 for k in CONTRACT}
    line["config"] = {f"key{i}": "some text of ordinary length" for i in range(12)}
    line["roofline"] = {k: 1.23456 for k in bench.SHORT["roofline"]} | {"evals_mean_by_n": {n: 1.0 for n in range(400)}}
    line["e2e"] = {"value": 2.0, "unit": "stencils/s", "h2d_bytes_per_step": 3, "d2h_bytes_per_step": 4,
                   "ms_per_step": [1.5] * 500}
    line["clocks"] = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}
    line |= {k: {"x": [1.0] * 3000} for k in bench.DETAILS}
    line["imex_step"] = {"ms": 1.7, "loop_iterations_per_step": [9] * 300}
    out = bench.short_line(line)
    assert all(k in out for k in CONTRACT)
    assert out["e2e"] == {"value": 2.0, "unit": "stencils/s", "h2d_bytes_per_step": 3, "d2h_bytes_per_step": 4}
    assert out["clocks"] == line["clocks"] and out["config"] == line["config"]
    assert len(json.dumps(out)) < 2500
    assert "x" in line["other_configs"]   # the details stay whole
