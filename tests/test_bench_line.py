"""The benchmark's printed line: every key of the measurement, the extra legs cut down to their figures of
merit, and short enough for a reader that keeps only the last few kilobytes of the output."""
import json

import bench


def _quantiles():
    return {k: 0.0012345678901234567 for k in ("mean", "p50", "p90", "p99", "max", "frac_le_tol")}


def _line():
    policy = {"ms": 3.1415926535897931, "speedup_vs_plain": 5.4321098765432101, "output": "Q on the grid (N^3 per cell)",
              "band_rel_l2_vs_fp32_plain": _quantiles(), "band_rel_l2_vs_fp64_first1024": _quantiles(),
              "full_Q_rel_l2_vs_plain_first1024": _quantiles()}
    names = ["checked_catch_all_to_grid", "checked_budget0.02_to_grid", "checked_budget0.04_to_grid", "checked_budget0.08_to_grid",
             "checked_budget_to_grid", "no_audit_unjudged", "audit_strict", "audit_tolerant"]
    kernel = {"plain_ms": 20.123456789, "policies": {n: dict(policy) for n in names}, "train": {"final_loss": 1e-6}}
    cfg = bench.workload_config(4096)
    cfg["shapes"] = [{"N": N, "cells": 1024, "cluster": 12, "threads": 288, "prefetch": 1, "tuned_us": 2345} for N in bench.N_CHOICES]
    return {"metric": bench.METRIC, "value": 2.2e10, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 10.3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic", "config": cfg,
            "cells_per_s": 4e5, "status": 0, "roofline": {"bound": "alu", "frac": 0.3}, "clocks": {"sm_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 1.5e10, "unit": bench.UNIT, "h2d_bytes_per_step": 917706752, "d2h_bytes_per_step": 918034432},
            "gpu_launches": 80, "surrogate": {"workload": "x" * 200, "kernels": {"hard_sphere": kernel, "maxwell": kernel}},
            "hbm_kernels": {k: {"cells": 4096, "ms": 0.1, "GBps": 6000.0, "frac_of_measured_hbm": 0.93} for k in ("moments_F", "transport")},
            "precision": {"config4": {"workload": "y" * 200, "fp32_ms": 40.0, "fp64_ms": 95.0, "errors": _quantiles()},
                          "config1": {"gpu_ms_per_step": 0.02, "oracle_ms_per_step": 0.3}},
            "cpu_baseline": {"value": 2300.0, "unit": bench.UNIT, "sample": "z" * 200}}


def test_line_is_short_and_complete():
    line = _line()
    assert len(json.dumps(line)) > 8000
    short, full = bench.printed_line(line)
    text = json.dumps(short)
    assert "\n" not in text and len(text) < 4500
    assert set(short) == set(line)
    for k in line:
        if k not in full:
            assert short[k] == line[k], k
    assert full == {k: line[k] for k in ("surrogate", "hbm_kernels", "precision")}
    assert short["surrogate"]["maxwell"]["speedup_vs_plain"]["checked_budget_to_grid"] == 5.4321
    assert short["hbm_kernels"] == {"moments_F": 0.93, "transport": 0.93}
    assert short["precision"]["config4"] == {"fp32_ms": 40.0, "fp64_ms": 95.0}


def test_a_failed_leg_keeps_its_reason_and_a_skipped_one_no_key():
    line = _line()
    line["hbm_kernels"] = {"error": "RuntimeError: " + "e" * 5000}
    del line["precision"]
    short, full = bench.printed_line(line)
    assert short["hbm_kernels"]["error"].startswith("RuntimeError") and len(json.dumps(short)) < 4500
    assert "precision" not in short and full["hbm_kernels"] == line["hbm_kernels"]
