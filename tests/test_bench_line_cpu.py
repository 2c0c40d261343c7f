"""The bench's one line stays short enough to be read whole: the forms go into it without
their tables, lists and texts (a record of the shape that the forms have, 16 KB)."""

import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def record():
    table = {f"class_{i}": 1234.567890123456 for i in range(12)}
    one = {"value": 6.441447246278681, "unit": "Newton solves/s", "ms_per_step": 465.7338460286458, "steps": 3,
           "converged": True, "iterations": [[284] * 8] * 3, "phase_ms_one_step": table, "launches_one_step": table,
           "roofline": dict(table, isolated=table), "kernels": {"spmv": table, "mas_apply_l0": table},
           "cpu_baseline": {"value": np.float64(0.03740310693206968), "cores": 8, "kind": "oracle", "sample": "x" * 400,
                            "host": {"nproc": 16}}, "workload": "y" * 300}
    return {"mixed": {k: dict(one) for k in "abc"}, "batched": dict(one), "newton": dict(one), "skipped": None,
            "differentiation": {"error": "z" * 300}}


def test_brief_keeps_the_rates_and_drops_the_tables():
    import bench

    full = record()
    out = bench.brief(full)
    text = json.dumps(out)  # plain numbers only
    assert len(text) < 2500 < 12000 < len(json.dumps(full, default=bench._json_scalar))
    a = out["mixed"]["a"]
    assert a["value"] == 6.4414 and a["unit"] == "Newton solves/s" and a["steps"] == 3 and a["converged"] is True
    assert a["cpu_baseline"] == {"value": 0.037403, "cores": 8, "kind": "oracle"}
    assert not {"roofline", "kernels", "iterations", "phase_ms_one_step", "workload"} & set(a)
    assert out["differentiation"]["error"] == "z" * 300 and "skipped" not in out
