"""The bench's stdout line stays short whatever its side sections hold, keeps
every key of the contract, and drops nothing but long sweeps."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline")


def test_line_is_short_and_keeps_the_contract():
    line = {k: {"value": 1.5} if k in ("config", "clocks", "e2e", "roofline") else k for k in CONTRACT}
    line["sweep"] = [dict({k: 0.123456789012345 for k in bench.SWEEP_KEYS}, extra="x" * 300) for _ in range(5)]
    for k in bench.SECTIONS:
        line[k] = {"workload": k, "mlups": 12345.678901234567, "timing": {"128": {"ms_per_step": 0.01}},
                   "sweep": [{"level": i, "threshold": 0.01, "ratio": 3.25} for i in range(400)]}
    line["swe"] = None
    full = json.dumps(line)
    out = bench.compact(line)
    assert len(full) > 60000 and len(json.dumps(out)) < 8000
    assert all(out[k] == line[k] for k in CONTRACT)
    assert out["swe"] is None and out["transport"]["timing"] == line["transport"]["timing"]
    assert all("sweep" not in out[k] for k in bench.SECTIONS if out[k]) and set(out["sweep"][0]) == set(bench.SWEEP_KEYS)
    assert json.dumps(line) == full
