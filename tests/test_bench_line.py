"""The line that bench.py prints stays short enough to be read whole, with the
keys of its contract, however much the record holds."""
import argparse
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _record(ncase):
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 12}
    roof = {"bound": "alu", "kernel": "k_fdpf_multi", "achieved": 0.5123456789, "peak": 1.2590123456, "unit": "TFLOP/s",
            "frac": 0.407123456, "traffic": 1.23456789e9, "peak_source": "FP64 unit count x SM clock (2 DFMA/cycle/SM x 152 SMs)",
            "algorithmic_fp64_flops_per_launch": 1.23456789e10, "kernel_ms_per_launch": 20.123456789,
            "hbm": {"bound": "hbm", "achieved": 123.456789, "peak": 6781.1, "unit": "GB/s", "frac": 0.0182, "peak_source": "measured",
                    "algorithmic_bytes_per_launch": 1.23456789e9}}
    acc = {"cases": ncase, "reference": "oracle Newton-Raphson to 1e-12 p.u., FP64", "max_dV_pu": 3.8123456e-10,
           "max_dtheta_rad": 3.6123456e-10, "median_dV_pu": 3.1e-10, "median_dtheta_rad": 3.2e-10, "worst_case": 17,
           "oracle_failed": 0, "per_case_dV_pu": [3.58e-10] * ncase, "per_case_dtheta_rad": [3.58e-10] * ncase,
           "seconds": 12.3456789, "cores": 16}
    cpu = {"value": 487.42324600118906, "unit": "PF/s", "cores": 16, "kind": "oracle",
           "sample": "5870 10k-bus cases (FP64 FDPF incl. ordering/symbolic/factor) across 16 processes in 12.0 s"}
    e2e = {"value": 158.93197711374572, "unit": "PF/s", "h2d_bytes_per_step": 80000, "d2h_bytes_per_step": 160024}
    config = {"workload": "plain10k", "nbus": 10000, "nbranch": 13500, "ncase": ncase, "ncase_per_rank": ncase,
              "precision": "fp64", "tol_pu": 1e-8, "ir_tol": 1e-3, "method": "fdpf", "engine": "auto",
              "l2": "flushed between timed steps (2.5x L2 buffer write)", "loading_factor": 0.03125, "analyze_ms": 30.2772,
              "tuning": {"engine": 1, "cluster": 16, "factor": 1, "tail": 3, "outage": 2, "threads": 512, "ms": 3.1234567,
                         "tune_s": 0.1234567}, "parallelism": "cases partitioned over 8 ranks"}
    kinds = ["ybus", "spec", "assemble", "factor", "solve", "mismatch", "run"]
    line = {"metric": "power-flow solves/s at 1e-8 pu mismatch", "value": 834.6123456789, "unit": "PF/s", "n_gpus": 1,
            "steps": 20, "warmup": 5, "ms_per_step": 1.19812345678, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "config": config, "converged": ncase, "ncase": ncase,
            "iters_mean": 17.123456, "iters_max": 20, "ir_steps_mean": 0.123456789, "ir_steps_max": 3, "gpu_launches": 360,
            "kernel_ms_per_step": {k: 1.23456789 for k in kinds}, "kernel_launches_per_step": {k: 2.0 for k in kinds},
            "cuda_graph": {"launches_per_step": 18.0, "ms_per_step_graph": 1.198, "ms_per_step_direct": 1.298},
            "roofline": roof, "clocks": clocks, "e2e": e2e, "cpu_baseline": cpu, "accuracy": acc}
    line["batched_fp32_ir"] = {k: line[k] for k in ("value", "unit", "ms_per_step", "dtype", "converged", "gpu_launches", "roofline",
                                                    "e2e", "clocks", "ir_steps_mean", "ir_steps_max", "iters_mean", "accuracy",
                                                    "cpu_baseline", "config")}
    return line


@pytest.mark.parametrize("ncase", [1, 1024])
def test_line_is_short_and_complete(ncase, capsys, tmp_path):
    sys.path.insert(0, ROOT)
    import bench
    record = _record(ncase)
    path = tmp_path / "record.json"
    bench.emit(record, argparse.Namespace(details=str(path)))
    text = capsys.readouterr().out.strip()
    assert len(text) <= bench.LINE_MAX and "\n" not in text
    d = json.loads(text)
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
              "clocks", "gpu_launches"):
        assert d[k] == record[k]
    for k in ("value", "ms_per_step"):
        assert abs(d[k] - record[k]) <= 1e-6 * record[k]
    assert set(d["e2e"]) == set(record["e2e"]) and d["e2e"]["h2d_bytes_per_step"] == 80000
    assert d["config"]["workload"] == "plain10k" and "l2" in d["config"] and "parallelism" in d["config"]
    assert d["batched_fp32_ir"]["value"] > 0 and d["accuracy"]["max_dV_pu"] > 0 and d["roofline"]["frac"] > 0
    with open(path) as fh:
        assert json.load(fh) == json.loads(json.dumps(record))
