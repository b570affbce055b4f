"""bench.py's printed line: one that a reader of the last few kilobytes of
output finds whole, whatever else a run measured."""

import json

import bench


def _record():
    mode = dict(ms_per_step=0.123456789, particles_per_s=1.234567890123e10,
                mean_path_len=1.6655512313, max_path_len=39, err_mean=0.00123456,
                err_vs_asg={"a": 1.0}, stages={"walk": 0.05, "cnn": 0.02})
    return {
        "metric": "particles located/s", "value": 13012345678.90123, "unit": "particles/s",
        "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 0.07678901234,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": bench.WORKLOADS["tg2d"]["desc"] + ", CFL 8",
                   "mode": "CNN-SNS (Algorithm 2)",
                   "particles": "one per mesh node, from the node's element",
                   "n_particles": 1002001, "n_elements": 2000000, "asg_grid": [1000, 1000],
                   "predictor_grid": {"stride": 5, "cells": [200, 200]},
                   "l2": "flushed by a 256 MB write before every timed step",
                   "parallelism": "8 replicas: every rank locates its own batch of 1002001 "
                                  "particles against its own copy of the mesh, no collective",
                   "arithmetic": "walk decisions FP64 (certified FP32 filter); predictor "
                                 "BF16 x BF16 -> FP32 on tcgen05"},
        "mean_path_len": 1.66555, "max_path_len": 39, "err_mean": 0.0012,
        "modes": {m: mode for m in ("sns", "asg", "cnn")}, "opt": {"x": [mode] * 20},
        "training": {"losses": [0.1] * 1000}, "classifier": {"rows": [mode] * 40},
        "serving": {"requests": [mode] * 40}, "sweep": [mode] * 60,
        "rooflines": {k: mode for k in "abcdef"},
        "roofline": {"bound": "hbm", "achieved": 2644.8672849189, "peak": 6786.2, "unit": "GB/s",
                     "kernel": "walk_kernel<2>", "kernel_ms": 0.0550032002851367,
                     "algorithmic_bytes_per_launch": 145476165.0, "traffic": None,
                     "peak_source": "measured", "frac": 0.38974},
        "cpu_baseline": {"value": 5903780.725553872, "unit": "particles/s", "cores": 16,
                         "kind": "oracle",
                         "sample": "1002001 of the 1002001 particles (seeded draw), the oracle's "
                                   "plain SNS: departure point + Algorithm 1 walk + exact host, "
                                   "its particle loops on 16 OpenMP threads, 0.17 s",
                         "single_core": {"value": 877083.79, "sample": "x" * 500}},
        "e2e": {"value": 4.6123456789e9, "unit": "particles/s", "h2d_bytes_per_step": 16032016,
                "d2h_bytes_per_step": 9018009, "entry_point": "cs_track_nodes_host",
                "transfer": "y" * 500, "general_call": {"value": 4.1e9, "transfer": "y" * 500}},
        "gpu_launches": 40,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"],
                   "samples": 61},
    }


def test_the_line_is_short_and_complete():
    full = _record()
    text = json.dumps(bench.headline(full))
    assert len(text) < bench.LINE_LIMIT <= 2500
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
              "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert k in line, k
    assert abs(line["value"] / full["value"] - 1) < 1e-5
    assert set(line["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert set(line["clocks"]) >= {"sm_mhz", "sm_max_mhz", "reasons"}
    assert line["config"] == full["config"]
    assert line["modes"]["sns"] == {"ms_per_step": 0.123457, "mean_path_len": 1.66555}


def test_parts_that_were_not_measured_are_left_out():
    full = _record()
    full["cpu_baseline"] = None
    full["clocks"] = None
    line = bench.headline(full)
    assert "cpu_baseline" not in line and line["clocks"] is None
