"""bench.py's result line: every headline key, short enough for a reader that keeps the
last 3,000 characters of a run's output."""
import json

import bench


def test_result_line_is_short_and_complete():
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 123}
    run = {"sweep_ms": 1000.123456789, "sweep_launches": 180}
    roof = bench._sweep_roofline_fp64(run, 256 ** 3, 7, "weno5", 2, clocks)
    kernels = {k: 123.45678901234567 for k in ("prims", "prims_cfl", "sweep_x", "sweep_y", "sweep_z", "cbc", "cons")}
    entry = {"grind": 0.0123456789012, "unit": bench.UNIT, "ms_per_step": 123.4567890123, "kernels_ms": kernels,
             "roofline": roof, "clocks": clocks, "config": {"notes": "n" * 400}}
    line = {"metric": bench.METRIC, "value": 0.0676543210987, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 23.8123456789, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic", "config": {"workload": "w" * 60, "arithmetic": "a" * 200, "l2": "l" * 60,
                                                            "cells": 16777216, "parallelism": "single-gpu"},
            "cell_updates_per_s": 7.0612345678e8, "roofline": roof, "gpu_launches": 180, "kernels_ms": kernels,
            "fallback_faces": 123456, "clocks": clocks,
            "forms": {f: entry for f in bench.FORMS if f != "fp64"}, "configs": {c: entry for c in bench.CONFIG_RUNS},
            "e2e": {"value": 0.102123456789, "unit": bench.UNIT, "h2d_bytes_per_step": 939524096,
                    "d2h_bytes_per_step": 939524096, "steps": 10, "note": "n" * 80},
            "cpu_baseline": {"value": 13.9, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 120,
                             "one_core": entry}}
    text = json.dumps(bench.summary(line))
    assert len(text) < 2800 and "\n" not in text
    out = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches", "e2e"):
        assert k in out
    assert abs(out["value"] - line["value"]) < 1e-6 and out["e2e"]["h2d_bytes_per_step"] == 939524096
    assert set(out["forms"]) == set(line["forms"]) and set(out["configs"]) == set(line["configs"])
