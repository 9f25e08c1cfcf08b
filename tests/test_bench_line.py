"""The line that the benchmark prints (and the DRAM figures in it): every key of the headline, and short -- a reader of the
last two kilobytes of output has it whole."""
import json

import bench
from test_bench_host import _fake_line


def full_line():
    line = dict(_fake_line(), metric="GLUPS", unit="GLUPS", n_gpus=1, steps=20, warmup=5, ms_per_step=7.123456789012,
                higher_is_better=True, scaling="weak", vs_baseline=None, dtype="f32", data="synthetic",
                status="VLBM_OK", gpu_launches=10, repeats=[1.0] * 5, slab_check=None,
                paper_context={"note": "x" * 200},
                clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 100},
                e2e={"value": 9.1, "unit": "GLUPS", "h2d_bytes_per_step": 214748364, "d2h_bytes_per_step": 214748368,
                     "runs_glups": [9.0, 9.1], "ms": {"steps": 1.0}, "note": "y" * 400},
                cpu_baseline={"value": 0.03, "unit": "GLUPS", "cores": 16, "kind": "oracle", "sample": "z" * 100})
    line["value"] = 18.361234567890123
    line["config"] = {"workload": bench.WORKLOAD, "grid": "512^3", "cells": 512 ** 3, "storage": "f32",
                      "populations_per_cell": 56, "parallelism": "single domain",
                      "l2": "inputs_larger_than_l2 (30.1 GB of populations per rank)"}
    line["roofline"] = {"bound": "hbm", "achieved": 4934.123456789, "peak": 6784.2, "unit": "GB/s",
                        "frac": 0.727312345678, "traffic": None, "kernel": bench.STEP_KERNEL["f32"]}
    line["summary"] = dict(bench.compact_summary(line), channel_u_err_5000=[0.6, 0.3, 0.08])
    return line


def test_printed_line_is_short_and_whole():
    line = full_line()
    out = bench.printed_line(line)
    assert len(json.dumps(out)) < 1900
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "gpu_launches", "status", "fp64_tflops"):
        assert out[key] == line[key]
    assert out["clocks"] == line["clocks"] and out["config"]["workload"] == bench.WORKLOAD
    assert out["e2e"] == {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert out["roofline"]["frac"] == line["roofline"]["frac"]
    assert out["paths"]["form_f16dev"] == [27.0, 0.9] and out["paths"]["channel"] == [20.5, 0.98]
    assert not any("_err_" in k for k in out["paths"])  # rates only
    assert json.loads(json.dumps(out)) == out


def test_printed_line_without_end_to_end():
    line = dict(full_line(), e2e=None, cpu_baseline=None)
    out = bench.printed_line(line)
    assert out["e2e"] is None and out["cpu_baseline"] is None


def test_traffic_of_two_step_passes_only_at_the_size_it_was_captured():
    one = bench.MEASURED_DRAM_BYTES_PER_CELL["f32"]
    two = bench.MEASURED_DRAM_BYTES_PER_CELL_TWO_STEPS["f32", 256]
    assert bench.dram_bytes_per_cell("f32", 512, 20, 0) == one
    assert bench.dram_bytes_per_cell("f32", 512, 10, 10) is None
    assert bench.dram_bytes_per_cell("f32", 256, 10, 10) == two
    assert abs(bench.dram_bytes_per_cell("f32", 256, 11, 9) - (2 * one + 9 * two) / 11) < 1e-9
    assert bench.dram_bytes_per_cell("f64", 512, 20, 0) is None
