"""The benchmark's one line of output: short enough for a reader that keeps the
last few kilobytes, with every figure of the headline in it."""
import argparse
import json

import bench


def _leg(value):
    return {"precision": "fp16_scaled", "arithmetic": bench.PREC_TEXT[3] + "; " + bench.SOLVE_TEXT,
            "ms_per_step": 1 / 3, "step_ms": [1 / 3] * 20, "tuning": {"k" * 60: list(range(9))},
            "autotune_s": 1 / 3, "kernels_ms": {k: 1 / 3 for k in ("doppler", "covariance", "solve", "apply")},
            "kernels_used": {"covariance": "tensor cores", "apply": "tensor cores"}, "value": value,
            "kernels": {k: {"a" * 40: 1 / 3, "b" * 40: 2 / 3} for k in ("doppler", "covariance", "solve", "apply")}}


def test_the_line_is_short_and_keeps_the_headline(tmp_path, capsys):
    value = 16777216 / 0.31
    errors = {lb: {"normwise": 4.03e-4 / 3, "max_cell": 0.07 / 3, "blocks": 8}
              for lb in ("fp16_scaled", "fp32", "fp16_scaled+mixed_ir")}
    cpu = {"value": 1e5 / 3, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "x" * 150}
    single = {"config": bench.workload_config(bench.workload_spec(0, "standard"), "standard"), "mixed": _leg(value),
              "fp32": _leg(value), "mixed_ir": _leg(value), "mixed_vs_fp32": 1 / 3, "errors_vs_oracle": errors,
              "cpu_baseline": cpu, "options": {k: _leg(value) for k in ("staggered", "neighbour_training",
                                                                       "window_training")}}
    cfg = bench.workload_config(bench.workload_spec(0, "large"), "large")
    cfg["precision"] = _leg(0)["arithmetic"]
    line = {"metric": bench.METRIC, "value": value, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 310 / 3, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "fp16+f32+f64", "data": "synthetic", "config": cfg,
            "e2e": {"value": value, "unit": bench.UNIT, "h2d_bytes_per_step": 1 << 32, "d2h_bytes_per_step": 1 << 32,
                    "ms_per_step": 1 / 3, "api": "x" * 220},
            "gpu_launches": 80, "mixed": _leg(value), "fp32": _leg(value), "mixed_ir": _leg(value),
            "mixed_vs_fp32": 1 / 3,
            "roofline": {"kernel": bench.SOLVE_KERNEL, "bound": "alu", "achieved": 40 / 3, "peak": 40.27392,
                         "unit": "T FP32 instructions/s", "frac": 1 / 3, "traffic": None, "basis": "x" * 400,
                         "fp64_equivalent_tflops": 10 / 3, "peak_src": "x" * 70},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 66},
            "errors_vs_oracle": errors, "cpu_baseline": cpu,
            "workloads": {"mixed": single, "standard": single, "batch": {"error": "x" * 100}}}
    path = tmp_path / "detail.json"
    bench.emit(line, argparse.Namespace(detail=str(path)))
    text = capsys.readouterr().out
    assert text.count("\n") == 1 and len(text) < 4000
    got = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert got[k] == line[k], k
    assert got["roofline"]["achieved"] == 13.3333 and got["kernels_ms"]["solve"] == 0.333333
    assert set(got["workloads"]["standard"]) == {"mixed", "fp32", "mixed_ir", "staggered", "neighbour_training",
                                                 "window_training"}
    assert got["workloads"]["batch"] == {"error": "x" * 100}
    with open(path) as f:
        assert json.load(f) == line
