"""The line that bench.py prints: every key of its contract, and a few KB however much the workloads
report."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches")


def record():
    sweep = {"row %d" % i: {"value": 1.0 / 3, "note": "x" * 40} for i in range(400)}  # some 35 KB
    out = {k: "text" for k in CONTRACT}
    out.update(value=6.5e8, vs_baseline=None, config={"workload": "w", "precision": "fp32"}, phases_ms={"m2l": 0.2},
               roofline={"frac": 0.5}, roofline_m2l=None, cpu_baseline={"value": 1e5}, peaks=sweep, operators=sweep,
               leaf_size=sweep, paper_shape=sweep, adaptive=sweep, batch=sweep, noalloc=sweep)
    out["modes"] = {m: {"value": 1e7, "ms_per_step": 100.0, "phases_ms": sweep, "rooflines": sweep}
                    for m in ("mixed", "fp64", "fp64_dense_m2l", "fp32_tf32_m2l", "ff")}
    rate = {"load": 0.5, "offered_solves_per_s": 1.0, "solves_per_s": 1.0, "particles_per_s": 1.0, "p50_ms": 1.0,
            "p99_ms": 1.0}
    out["serving"] = {"workload": "w", "saturated": {"solves_per_s": 1.0, "particles_per_s": 1.0, "p50_ms": 1.0,
                                                     "p99_ms": 1.0}, "rates": [rate] * 3, "accuracy": sweep}
    out["accuracy"] = {"rel_l2_phi_vs_oracle": 1e-6, "fp64_rel_l2_phi_vs_direct_by_order": {"p2": 1.0},
                       "smallest_order_reaching_1e-7": None}
    return out


def test_line_is_complete_and_short():
    out = record()
    assert len(json.dumps(out)) > 100_000
    text = json.dumps(bench.headline(out))
    line = json.loads(text)
    assert "\n" not in text and len(text) < 4096
    for k in CONTRACT:
        assert line[k] == out[k], k
    assert line["roofline"] == out["roofline"] and line["cpu_baseline"] == out["cpu_baseline"]
    assert line["modes"]["ff"] == {"value": 1e7, "ms_per_step": 100.0}
    assert line["served"]["p99_ms"] == 1.0 and len(line["served"]["rates"]) == 3
    assert line["accuracy"]["rel_l2_phi_vs_oracle"] == 1e-6


def test_line_without_the_extra_workloads():
    out = {k: v for k, v in record().items() if k in bench.HEADLINE_KEYS}
    line = bench.headline(out)
    assert line["value"] == out["value"] and "served" not in line and line["modes"] == {}
