"""The result line of bench.py: one short JSON line on stdout that keeps what it
has to report, whatever the detail sections hold.  CPU only."""
import json

import bench

REQUIRED = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
            "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
            "clocks", "gpu_launches")


def test_line_is_short_and_complete():
    details = {"n": list(range(2000)), "solves_per_s": 1000.5, "p50_ms": 1.5, "p99_ms": 9.5,
               "rate_0.8": {"p50_ms": 1.5}}
    line = {k: 1 for k in REQUIRED}
    line["config"] = {"workload": bench.WORKLOAD, "parallelism": "1 GPU"}
    line["roofline"] = {"frac": 0.9, "kernel": "k_ell"}
    line["cpu_baseline"] = None
    for k in bench.DETAILS:
        line[k] = details
    full = json.dumps(line)
    out = bench.headline(json.loads(full))
    text = json.dumps(out)
    assert len(full) > 50_000 and len(text) < 3000 and "\n" not in text
    assert all(out[k] == line[k] for k in REQUIRED)
    assert out["roofline"] == line["roofline"]
    assert out["cg"] == {"solves_per_s": 1000.5}
    assert out["serving"] == {"solves_per_s": 1000.5, "p50_ms": 1.5, "p99_ms": 9.5}
    line["cg"] = line["serving"] = None  # switched off
    assert "cg" not in bench.headline(line) and "serving" not in bench.headline(line)
