"""The default bench run prints one line that fits what keeps the end of its
output (3000 characters)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _record():
    import bench
    kernel = {"kernel": "k" * 90, "bound": "hbm", "achieved": 3456.7891, "peak": 6781.1, "unit": "GB/s", "frac": 0.5098,
              "traffic": {"dram_bytes": 141500000}, "peak_source": "measured copy", "algorithmic_bytes_per_launch": 141500000,
              "what": "w" * 60, "avg_launch_us": 41.23, "launches": 6900}
    rec = {"metric": bench.METRIC, "value": 19.9012, "unit": "solves/s", "n_gpus": 1, "steps": 20, "warmup": 5,
           "ms_per_step": 50.249, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64",
           "data": "synthetic",
           "config": {"workload": bench.WORKLOADS["ball1m"]["desc"], "n_cells": 1000000, "edges": 2363456,
                      "mean_degree": 4.727, "form": "mixed precision, tree preconditioner", "tol": 1e-08,
                      "step": "collision graph + friction blocks + spanning forest + tree factor + PCG solve",
                      "l2": "working set > L2 (friction blocks alone 359 MB: FP64 and FP32 records)", "parallelism": "single"},
           "iterations": 345, "true_rel_residual": 4.912345678901234e-09, "outer_iterations": 3,
           "solve_only": {"value": 23.6012, "unit": "solves/s", "ms_median": 42.412},
           "e2e": {"value": 19.5612, "unit": "solves/s", "h2d_bytes_per_step": 56000000, "d2h_bytes_per_step": 24000000,
                   "steps": 20},
           "gpu_launches": 12345, "roofline": kernel, "roofline_other": [kernel] * 9,
           "solve_roofline": {"frac": 0.6123, "bytes": 10 ** 11}, "tree_layout": {"bins": 0}, "time_share_ms": {"note": "n" * 90},
           "forms": {"plain_fp64_mst": {"solves_per_s": 6.9412, "iterations": 318}, "chosen_vs_plain_fp64": 2.867,
                     "fp64_block_jacobi": {"solves_per_s": 1.9112, "iterations": 1743}},
           "tuning": {}, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["gpu_idle"], "samples": 99},
           "cpu_baseline": {"value": 0.013712, "unit": "solves/s", "cores": 1, "kind": "oracle", "extrapolated": True,
                            "sample": "s" * 300, "all_cores": {"value": 0.021012, "unit": "solves/s", "cores": 16}}}
    rec["configs"] = {k: {"value": 1389.1234, "unit": "solves/s", "ms_per_step": 368.123, "forms": ["x" * 500]}
                      for k in ("cube1k", "hex4m", "batch512", "warm200k", "aug1m", "paper")}
    rec["configs"]["local1m"] = {"error": "e" * 400}
    return rec


def test_headline_is_short_and_keeps_the_contract():
    import bench
    rec = _record()
    line = bench.headline(rec)
    assert len(json.dumps(line)) <= 2900 < len(json.dumps(rec))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert line[k] == rec[k], k
    assert set(line["configs"]) == set(rec["configs"]) and line["configs"]["hex4m"]["value"] == 1389.1234
