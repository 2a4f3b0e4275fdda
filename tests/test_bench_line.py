"""The JSON line of bench.py: every key of the contract, and short enough that the last 3000 characters of
the output hold all of it (a longer line was cut and could not be read)."""
import argparse
import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

X = 12345678.901234567


def _form(form):
    kernels = ["k_fof_link", "k_sort_hist", "k_sort_scatter", "k_nn6d_pruned", "k_link6d_pruned", "k_tree_walk",
               "k_potential", "k_potential_blocked", "k_potential_list"]
    return {"form": form, "value": X * 20, "ms_per_step": X / 1e4, "steps": 20, "warmup": 5, "launches": 123456,
            "launches_per_step": X, "prof": {k: (X / 1e5 + i, 999) for i, k in enumerate(kernels)},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0,
                       "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_power_cap", "sw_thermal_slowdown"],
                       "samples": 1000},
            "fallback": 12345, "work": {"nn_d6": 1 << 40, "link_d6": 1 << 40}, "n": 1 << 27, "members": 118627377,
            "nodes": 655360, "digest": "0" * 64, "tree": {"expansions": 1 << 40, "direct_pairs": 1 << 40, "list_pairs": 1 << 40},
            "surrogate_stats": {}, "sort_keypasses": 1 << 33, "autotune": {}, "bound_host": np.zeros(10, np.uint8),
            "pairs": {"pairs_all": X * 1e6, "pairs_small": X * 1e3, "pairs_blocked": X * 1e4}}


def test_line_is_short_and_complete():
    res = {f: _form(f) for f in ("surrogate", "batched", "surrogate_calibrated", "plain")}
    args = argparse.Namespace(steps=20, warmup=5, workload=bench.DEFAULT_WORKLOAD)
    cpu = {"value": X / 50, "unit": bench.UNIT, "cores": 144, "kind": "oracle", "sample": "s" * 200}
    e2e = {"value": X * 20, "unit": bench.UNIT, "h2d_bytes_per_step": 1 << 32, "d2h_bytes_per_step": 1 << 31, "steps": 20}
    stream = {"particles": 1 << 27, "sequential": {"value": X * 15}, "lanes": {"value": X * 30}, "identical_outputs": True}
    line, details = bench.result_lines(args, res, 8, 1 << 27, 512.0, 3, {}, cpu, e2e, {"train_s": X}, stream)
    text = json.dumps(line)
    assert len(text) <= 2000, len(text)
    assert "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in line, key
    assert line["value"] == X * 20 and line["ms_per_step"] == X / 1e4
    assert set(line["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert line["e2e"]["value"] == float(f"{X * 20:.9g}")
    assert line["flag_mismatches"] == 0 and line["identical_outputs"] is True
    assert set(details["forms"]) == set(res) and json.dumps(details)
    assert bench.result_lines(args, {"surrogate": res["surrogate"]}, 1, 1 << 27, 512.0, 3, {}, None, e2e, None, None)[0][
        "flag_mismatches"] is None
