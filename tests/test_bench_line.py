"""The line that the bench prints stays short however much its record holds, and keeps every key its readers need."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "cpu_baseline", "roofline")


def _record():
    surface = {f"R_{i}": 1.0 / (i + 3) for i in range(12)}
    stage = {"mean_tflops": 1 / 3, "p50_tflops": 1 / 3, "p99_tflops": 1 / 3, "R_N_slice": 1 / 3, "R_3D": 1 / 3,
             "roofline_mean_frac": 1 / 3, **surface}
    text = "x" * 480
    return {"metric": bench.METRIC, "value": 795.123456789, "unit": "TFLOP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 9600.123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic",
            "config": {"workload": text[:150], "smoothed": text[:250], "plain": "fixed 128x128 tile, split 1", "timing": text,
                       "parallelism": "single GPU"},
            "plain": stage, "smoothed": stage, "roughness_cut_pct": 6.2, "mean_gain_pct": 21.0,
            "roofline": {"bound": "tensor", "achieved": 1426.123456, "peak": 1948.6, "unit": "TFLOP/s", "frac": 0.7318888,
                         "traffic": None, "traffic_note": text, "mean_frac": 0.4494444, "kernel": "gemm_bf16 256x256/2SM",
                         "note": text},
            "roofline_capture": {"bound": "tensor", "kernel": text[:80], "shape": [8192, 8192, 4096], "achieved": 1.1,
                                 "frac": 0.9, "traffic": 1, "algorithmic_bytes": 2, "note": text},
            "roofline_all_gemms": {"achieved": 1400.1, "frac": 0.72, "unit": "TFLOP/s"},
            "peak_cell": {"M": 1, "N": 2, "K": 3, "tflops": 1.5, "variant": "256x256/2SM", "frac": 0.9},
            "gpu_launches": 1390000, "sm_count": 152, "setup_s": 289.1,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 900, "reasons": ["sw_power_cap"]},
            "e2e": {"value": 61.0178, "unit": "TFLOP/s", "h2d_bytes_per_step": 1554382848, "d2h_bytes_per_step": 1739522048,
                    "api": "rg_gemm_plan_host (C ABI, host buffers)", "sample": text},
            "cpu_baseline": {"value": 0.59, "unit": "TFLOP/s", "cores": 16, "kind": "oracle", "cpu_model": "Neoverse-V2",
                             "blas": {"name": "openblas", "version": "0.3.34", "openblas configuration": text},
                             "sample": text, "small_sweep_64_cells": {"a": 1}},
            "ladder": {f"stage{i}": stage for i in range(40)}, "surface": [1.23456789] * 4096}


def test_line_is_short_and_complete():
    record = _record()
    line = bench.short_line(record)
    printed = json.dumps(line)
    assert len(printed) <= bench.LINE_BYTES and "\n" not in printed
    assert all(k in line for k in CONTRACT)
    assert line["value"] == record["value"] and line["ms_per_step"] == record["ms_per_step"]
    assert line["e2e"]["h2d_bytes_per_step"] == 1554382848 and line["e2e"]["value"] == 61.0178
    assert line["clocks"] == record["clocks"] and line["config"] == record["config"]


def test_line_without_extras():
    record = {k: v for k, v in _record().items() if k not in ("e2e", "cpu_baseline", "ladder", "roofline_capture")}
    line = bench.short_line(record)
    assert "e2e" not in line and line["plain"]["mean_tflops"] == 0.333333
