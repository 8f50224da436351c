"""bench.py's line on standard output: every key of its contract, whole in the last 3,000 characters of a log."""
import json

import bench

KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
        "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches")


def record():
    x = 1234.5678901234567
    full = {k: x for k in bench.LINE_KEYS}
    full.update(vs_baseline=None, metric=bench.METRIC)
    cfg = {"variant": 0, "ctas_per_sm": 3, "grid_mult": 8, "batch": 128, "min_blocks": 3, "occupancy": 3}
    full["config"] = {"workload": bench.WORKLOAD, "l2": "x" * 80, "launch": {"pose_grad": cfg, "forward": cfg},
                      "evaluations": 265145319, "pair_pixels": 265361536, "blended": 38639568}
    full["clocks"] = {"sm_mhz": x, "sm_max_mhz": x, "reasons": [], "window": "x" * 80}
    full["e2e"] = {"value": x, "unit": "Mpix/s", "ms_per_step": x, "h2d_bytes_per_step": 33177600,
                   "d2h_bytes_per_step": 56, "transfer": "x" * 120}
    full["roofline"] = {"bound": "alu", "achieved": x, "frac": x, "work": "x" * 200}
    full["kernels"] = {k: {"ms": x, "share": x} for k in ("project", "shade", "scan_tiles", "scatter", "sort")}
    full["untuned"] = {"ms_per_step": x, "note": "x" * 60}
    full["cpu_baseline"] = {"value": x, "unit": "Mpix/s", "cores": 16, "kind": "oracle", "sample": "x" * 400}
    full["pmm"] = {"ms": x, "decisions": {"x": ["x" * 100] * 10}}
    full["errors"] = {"outputs": ["x" * 100] * 100}
    return full


def test_short_line_holds_the_contract_and_fits():
    full = record()
    line = bench.short_line(full)
    assert len(json.dumps(line)) <= bench.LINE_LIMIT <= 2900
    for k in KEYS:
        assert line[k] == full[k], k
    assert line["sections"]["match_ms"] == float("%.5g" % full["pmm"]["ms"])
    assert "errors" not in line and len(json.dumps(full)) > 10000


def test_short_line_without_optional_sections():
    full = {k: 1 for k in KEYS}
    line = bench.short_line(dict(full, refine=None, pmm=None, cpu_baseline=None))
    assert {k: line[k] for k in KEYS} == full
