"""CPU test of the benchmark's output: one JSON line, short enough to survive a
log that keeps the last 3000 characters, with the side legs summarised."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

F = 1234567890123.4567  # as many digits as a float has


def _line():
    """A line with every leg, as long as the default run makes it."""
    load = {"p50_ms": F, "p99_ms": F, "pairs_per_s": F, "jobs_per_s": F, "makespan_s": F}
    modes = {m[0]: {"ms": F, "eta": F, "max_rel_err": F} for m in bench.TABLE6_MODES}
    method = {"time_s": F, "iters": 300, "sse": F, "ami": F, "ari": F, "diff_vs_fp64": 0.0, "eta": F, "speedup_vs_fp64": F}
    methods = {m: dict(method) for m in ("FP64", "FP32", "BF16->FP64 rho=5", "FP16->FP64 rho=5", "FP16->FP64 rho=50")}
    return {
        "metric": bench.METRIC, "value": F, "unit": "pairs/s", "n_gpus": 1, "steps": 200, "warmup": 5, "ms_per_step": F,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": "c2a: " + bench.WORKLOADS["c2a"][4], "n": 1000000, "d": 128, "k": 1024, "low": "bf16",
                   "test": "tc", "rho": 5.0, "parallelism": "single", "step": 100 * "s", "l2": 60 * "l"},
        "roofline": {"bound": "tensor", "achieved": F, "peak": F, "unit": "TFLOP/s", "frac": F, "traffic": F,
                     "kernel": "k_tc (tcgen05 screen)", "algorithmic_flops_per_launch": F, "peak_source": 60 * "p"},
        "cpu_baseline": {"value": F, "unit": "pairs/s", "cores": 16, "kind": "oracle", "sample": 90 * "s", "seconds": F},
        "e2e": {"value": F, "unit": "pairs/s", "h2d_bytes_per_step": 512524288, "d2h_bytes_per_step": 12532480,
                "ms_per_step": F, "call": "km_lloyd_step_host"},
        "gpu_launches": 3400, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 99},
        "fp64_path": {"value": F, "unit": "pairs/s", "sample_rows": 65536, "repeats": 5, "ms_per_call": [F] * 5,
                      "labels_equal_on_sample": True, "mixed_over_fp64": F},
        "serving": {"jobs": 200, "iterations_per_job": 25, "arena_gb": 80, "saturated": load, "sizes": 90 * "s",
                    "formats": {"e4m3": 27}, "poisson_50%": load, "poisson_80%": load},
        "table6": {"n": 5000, "modes": {f: dict(modes) for f in ("near_0%", "near_10%", "near_50%", "near_90%")}},
        "quality": {"tau": 1e-8, "blobs": {"n=100000 d=%d k=%d" % (d, k): methods for d in (10, 128) for k in (100, 500)},
                    "image": {"1024x1024 d=5 k=%d" % k: methods for k in (8, 32)}},
        "c3_trajectory": {low: {"time_s": F, "iters": 50, "sse": [F] * 51, "labels_equal_fp64": True,
                                "max_rel_sse_diff_vs_fp64": F, "eta_mean": F} for low in ("fp64", "fp32", "bf16", "fp16", "e4m3")},
        "autotune": {"variant": "half", "ms_per_assign": {"full": F, "half": F, "c32": F}},
        "phases_ms_per_step": {p: F for p in ("quantise", "screen", "refine", "fullrow", "update", "direct")}, "eta": F,
        "assign_stats": {"fp32_evals": 2371533, "fp64_evals": 832, "ambiguous_rows": 416, "overflow_rows": 1000000},
    }


def test_the_line_fits():
    text = json.dumps(bench.compact(_line()))
    assert len(text) < 2800
    line = json.loads(text)
    assert set(line) == set(_line())
    assert abs(line["value"] / F - 1) < 1e-6 and line["e2e"]["h2d_bytes_per_step"] == 512524288
    assert line["c3_trajectory"]["labels_equal_fp64"] is True and "sse" not in json.dumps(line["quality"])


def test_skipped_and_failed_legs_pass_through():
    line = dict(_line(), serving=None, table6=None, quality={"error": "ValueError: x"}, c3_trajectory=None)
    got = bench.compact(line)
    assert got["serving"] is None and got["quality"] == {"error": "ValueError: x"} and got["c3_trajectory"] is None
