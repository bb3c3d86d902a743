"""The line that bench.py prints (no GPU): the contract's keys as they were measured, and short."""

import json

import bench

ITERS = [141, 141, 143, 146, 151, 131, 130, 131]


def _record():
    launch = {"us": 77.631, "us_median": 77.7, "us_min": 74.62, "gbs": 5609.123456, "frac_of_measured_peak": 0.826212, "alg_mb": 435.4,
              "tuned": {"m": 1, "dtype": "f64", "lanes": 1, "share": 32, "untiled": True, "best_us": 71.54}}
    solve = {"solves_per_s": 25.0212345, "seconds": 0.3197, "iters": ITERS, "outer": ITERS, "speedup_vs_one_rhs_f64": 2.3641234,
             "max_rel_err_vs_oracle": 9.36123e-06}
    served = {"p50_ms": 119.23456, "p99_ms": 1531.0, "requests_per_s": 2.94, "batch_cols_hist": {str(k): 100 for k in range(32)}}
    widths = [str(m) for m in bench.M_SWEEP]
    return {
        "metric": bench.METRIC, "value": 3532.123456789, "unit": "GB/s", "n_gpus": 1, "steps": 1500, "warmup": 5, "ms_per_step": 1.8234567891,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": {"n": 4194304},
        "roofline": {"frac": 0.42345678}, "sweep": {m: launch for m in widths}, "e2e": {"value": 310.71234567, "h2d_bytes_per_step": 2113929216},
        "cusparse_spmm": {m: {"us": 1054.0, "us_per_algorithm": {"a": 1.0}, "ours_speedup": 11.35} for m in widths},
        "solves": {w: {f"solver{k}": solve for k in range(12)} for w in ("a", "b")}, "cubes_gspmv": {"workload": "c", "sweep": {m: launch for m in widths}},
        "batch": {"rhs_solves_per_s": 50.31, "systems": [{"grid": "g" * 200}] * 4}, "serving": {**served, "whole_stream": served},
        "paper_estimate": {"rows": [{"k": 1.0}] * 100}, "cpu_baseline": {"value": 86.34, "kind": "oracle", "host": {"nproc": 16}},
        "clocks": {"sm_mhz": 2070.0}, "gpu_launches": 9000,
    }


def test_line_is_short_and_keeps_the_contract():
    r = _record()
    line = bench.short_line(r)
    assert len(json.dumps(r)) > 12000 and len(json.dumps(line)) < 5000
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
              "config", "roofline", "e2e", "clocks", "gpu_launches"):
        assert line[k] == r[k]
    assert line["sweep"]["32"] == {"us": 77.63, "gbs": 5609.0, "frac_of_measured_peak": 0.8262}
    assert line["solves"]["b"]["solver3"] == {"solves_per_s": 25.02, "max_rel_err_vs_oracle": 9.361e-06}
    assert line["cpu_baseline"] == {"value": 86.34, "kind": "oracle"} and line["serving"]["whole_stream"]["p99_ms"] == 1531.0
