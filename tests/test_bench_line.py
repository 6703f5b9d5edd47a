"""The benchmark's stdout line: short enough for a launcher that keeps the end of
the output, with every key of its contract, whatever the full result holds."""
import json

import pytest

import bench


def _full():
    row = {f"closest/kind{k}/cap3/dynamic_vs_static": 1.2345 for k in range(300)}
    return {
        "metric": bench.METRIC, "value": 12345.67, "unit": "Mrays/s", "n_gpus": 1, "steps": 20,
        "warmup": 5, "ms_per_step": 0.8123, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": bench.WORKLOAD, "rays_per_step": 4147200, "triangles": 1000002,
                   "launch": "params NULL, tuned on the frame before the steps",
                   "primary": "block=64 persistent=1 refill=24 stack_regs=0 image_width=1920 "
                              "ray_order=1 lockstep=1 octant=1",
                   "shadow": "block=64 persistent=1 refill=24 stack_regs=0 image_width=1920 "
                             "ray_order=1 lockstep=1 octant=1",
                   "l2": "flushed between steps (256 MiB write)",
                   "parallelism": "replicas x1 (each rank traces its own frame)"},
        "roofline": {"bound": "l1", "achieved": 28888.8, "peak": 40279.0, "unit": "GB/s",
                     "frac": 0.7172, "kernel": "trace closest alpha (primary)", "traffic": 1,
                     **row},
        "gpu_launches": 60, "breakdown": row, "large": row,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 40},
        "e2e": {"value": 4499.99, "unit": "Mrays/s", "h2d_bytes_per_step": 66355200,
                "d2h_bytes_per_step": 66355200, "bands": 8, "schedule": "x" * 300},
        "fwd_bwd": {"value": 1589.0, "unit": "Mrays/s", **row},
        "cpu_baseline": {"value": 13.7, "unit": "Mrays/s", "cores": 16, "kind": "oracle",
                         "sample": "x" * 200}}


def test_line_is_short_and_complete():
    out = _full()
    line = bench.headline(out)
    assert len(line) <= bench.LINE_LIMIT and "\n" not in line
    got = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
                "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "gpu_launches"):
        assert got[key] == out[key]
    assert got["config"]["workload"] == bench.WORKLOAD and "flushed" in got["config"]["l2"]
    assert got["e2e"] == {k: out["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step",
                                                     "d2h_bytes_per_step")}
    assert got["clocks"] == {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}
    out["config"]["workload"] = "x" * 3000
    with pytest.raises(ValueError, match="characters"):
        bench.headline(out)


def test_line_without_the_optional_parts():
    out = _full()
    for key in ("fwd_bwd", "cpu_baseline"):
        del out[key]
    out["clocks"] = None  # no sampler
    got = json.loads(bench.headline(out))
    assert got["clocks"] is None and "fwd_bwd" not in got
