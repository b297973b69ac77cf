"""The benchmark's result line stays short and keeps its contract's keys."""
import json

import bench


def _record():
    path = {"patterns_per_s": 1234567.123456789, "ms_per_step": 12.3456789, "steps": 10, "patterns_timed": 262144,
            "ms_per_timed_step": 12.3, "warmup": 3, "clocks": {"sm_mhz": 2070.0}, "launches_per_step": 56.0,
            "stages": {k: {"ms_per_step": 1.23456789, "launches_per_step": 14.0}
                       for k in ("polar", "prefilter", "sparse", "dft", "dense", "gemm", "select", "rescore")},
            "roofline": {"notes": "x" * 700}, "polar_roofline": {"notes": "x" * 700},
            "top1_vs_oracle": {"all": {"rate": 1.0}, "per_library": [{"rate": 1.0}] * 3}}
    return {"patterns": 262144, "libraries": [13986] * 3, "notes": "x" * 2000,
            "paths": {"fp32": path, "bf16": dict(path), "other": {"unsupported": "odd grid"}}}


def test_result_line_is_short():
    keys = ("metric value unit n_gpus steps warmup ms_per_step higher_is_better scaling vs_baseline dtype data config "
            "clocks e2e gpu_launches roofline cpu_baseline serving p99_line_ms two_stage preprocess").split()
    line = {k: {"notes": "x" * 150} for k in keys}
    line["workloads"] = {w: _record() for w in ("large_map", "multiphase", "single_phase")}
    line["paths"] = line["workloads"]["large_map"]["paths"]
    out = bench.compact_line(line)
    assert set(keys) <= set(out) and len(json.dumps(out)) < 8000 < len(json.dumps(line))
    fp32 = out["workloads"]["multiphase"]["paths"]["fp32"]
    assert fp32["patterns_per_s"] == 1234567.123456789 and fp32["top1_vs_oracle"] == 1.0
    assert out["workloads"]["large_map"]["paths"]["other"] == {"unsupported": "odd grid"}
