"""The benchmark's output line: every required key, short enough to be kept whole.

A caller keeps the last few thousand characters of the output; the line with the
autotuner's and the levels' tables was 22,000 characters long and was lost.
"""
import json

import bench


def _tables():
    rows = [{"level": l, "n_free": 10 ** l, **{f"stage{i}_ms": 0.123456789012345 for i in range(8)}} for l in range(8)]
    part = {"mixed_ms": 20.08675231933594, "mixed_iterations": 8, "fp64_ms": 53.48873519897461, "fp64_iterations": 8,
            "mixed_per_level": rows, "fp64_per_level": rows}
    x = 0.1234567890123456
    return {
        "metric": "fine-level vmult GDoF/s; solve time to 1e-8 rel. res., mixed/learned vs FP64", "value": 173.721200810325,
        "unit": "GDoF/s", "n_gpus": 8, "steps": 20, "warmup": 5, "ms_per_step": 20.086752319335936,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32 V-cycle / f64 CG",
        "data": "synthetic",
        "config": {"workload": "Q4 cube octant global5+2 (296,535 cells)", "degree": 4, "cells": 296535,
                   "n_free": 18740987, "levels": 8, "rhs": "8 Fourier modes, seed 2203", "rtol": 1e-08,
                   "l2": "inputs larger than L2 (finest level vectors and metadata > 129 MB)",
                   "parallelism": "replicas x8"},
        "roofline": {"bound": "hbm", "achieved": 1702.4677679411855, "peak": 6781.1, "unit": "GB/s", "frac": x,
                     "traffic": 257900000.0, "peak_kind": "measured", "alu_frac": x, "kernel": "k" * 200,
                     "traffic_source": "t" * 200},
        "alu_peaks": {"fp32_tflops": 78.5, "how": "h" * 100},
        "vcycle": {"ms": x, "gdofs": x, "frac": x, "what": "w" * 100},
        "cpu_baseline": {"value": x, "unit": "GDoF/s", "cores": 1, "kind": "oracle", "sample": "s" * 200},
        "e2e": {"value": x, "unit": "GDoF/s", "h2d_bytes_per_step": 74963948, "d2h_bytes_per_step": 74963948,
                "one_vector_per_call_gdofs": x, "call": "c" * 200},
        "gpu_launches": 123456,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 3, "samples_total": 12},
        "solve": {"mixed_ms": x, "mixed_iterations": 8, "mixed_rel_residual": 8.000095683052748e-10, "fp64_ms": x,
                  "fp64_iterations": 8, "fp64_rel_residual": 7.999978773308282e-10,
                  "solution_rel_diff_mixed_vs_fp64": 1.5264782938661885e-13, "fp64_arithmetic": "a" * 100},
        "vmult": {"fp32_ms": x, "fp32_gdofs": x, "fp64_ms": x, "fp64_gdofs": x, "fp64_hbm_frac": float("nan")},
        "configs": {"q2_octant": part, "q4_sphere_p": part}, "stage_ms_per_step_finest": rows[0],
        "coarser_levels_ms_per_step": x, "per_level_ms_per_step": rows, "setup_s": x,
        "learned": {"kept": "chebyshev",
                    "variants": [{"name": n, "ms": 41.02995300292969, "iterations": 14}
                                 for n in ("chebyshev", "augment", "replace")]},
        "batch": {"problems": 256, "dofs": 178707769, "solve_ms": x, "all_converged": True,
                  "tuning_candidates": {str(k): rows * 2 for k in (1, 2, 3, 4)},
                  "persistent": {"solve_ms": x, "all_converged": True, "max_rel_diff_vs_graph_batch": 8.5e-12,
                                 "solve_ms_all": [x] * 3}},
    }


def test_line_is_short_and_complete(tmp_path, monkeypatch, capsys):
    monkeypatch.setattr(bench, "__file__", str(tmp_path / "bench.py"))
    res = _tables()
    assert len(json.dumps(bench.finite(res))) > 10000
    bench.report(res)
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) <= bench.LINE_MAX
    line = json.loads(out)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "solve", "vmult"):
        assert key in line, key
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
    assert {"sm_mhz", "sm_max_mhz", "reasons"} <= set(line["clocks"])
    assert abs(line["value"] / res["value"] - 1) < 1e-5
    details = json.loads((tmp_path / bench.DETAILS).read_text())
    assert details["batch"]["tuning_candidates"]["4"] and details["per_level_ms_per_step"]
    assert details["vmult"]["fp64_hbm_frac"] is None


def test_parts_left_out():
    res = dict(_tables(), configs=None, learned=None, batch=None)
    line = bench.headline(bench.finite(res))
    assert "batch" not in line and "learned" not in line and line["value"]
