"""The benchmark's printed line: the contract's keys whole, and short enough to be
read back from a log (the full figures, tens of kilobytes, go to a file)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def _full(steps):
    stats = {c: {"ms": 12.3456789, "launches": 245, "flops": 4.1e11, "bytes": 6.3e9}
             for c in ("assemble", "diag", "trsm", "update", "update_tc", "queue")}
    mode = {"ms_per_step": 46.123456789, "step_ms": [46.123] * steps, "factor_ms": 28.01, "solve_ms": 17.9,
            "factor_bytes": 1444123456, "factor_gflops": 14800.1, "time_to_solve_gflops": 9007.123456,
            "backward_error": 1.4180053542798534e-13, "host_backward_error": 1.4180053542798534e-13,
            "rel_diff_to_fp64_solution": 1e-12, "refine_iters": 3, "converged": True, "launches_per_step": 1668,
            "e2e_ms": 47.8, "e2e_backward_error": 1.4e-13, "kernel_stats": stats,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 9}}
    point = {"N": 64, "M": 512, "us_per_call": 12.345, "gflops": 12345.6789, "gbs": 1234.56789}
    work = {"workload": "a description " * 8, "per_step": [1.0] * steps, "forward_ms": 22.0, "backward_ms": 50.2,
            "selected_inverse_ms": 47.4, "fp32_refined": {"ms": 26.3}, "fp64": {"ms": 70.6},
            "modes": {m: {"ms_per_step": 49.123456} for m in ("fp64", "fp32", "tf32", "bf16")},
            **{f"figure_{k}": 1234.56789 for k in range(12)}}
    modes = ("fp64", "fp32", "tf32", "bf16")
    return {"metric": bench.METRIC, "value": 9007.123456789, "unit": "GFlop/s", "n_gpus": 1, "steps": steps,
            "warmup": 5, "ms_per_step": 46.03, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": bench.DTYPES["tf32"], "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "n": 262144, "l2": "flushed between timed steps " * 3},
            "modes": {m: dict(mode) for m in modes}, "kernel_stats": {m: stats for m in modes},
            "fp64_ms_per_step": 84.5, "speedup_mixed_over_fp64": 1.84,
            "roofline": {"bound": "alu", "achieved": 12.3, "peak": 1258.0, "unit": "GFLOP/s", "frac": 0.01,
                         "kernel": "potrf_mid_kernel", "device_ms": 16.0},
            "rooflines": {c: dict(stats["diag"]) for c in stats}, "cpu_baseline": {"value": 2.5, "cores": 1},
            "e2e": {"value": 8676.1, "unit": "GFlop/s", "h2d_bytes_per_step": 48000000, "d2h_bytes_per_step": 33554432},
            "gpu_launches": 29000, "clocks": mode["clocks"], "update_kernel_study": {"points": [point] * 90},
            "batched_lu": work, "differentiation": work, "ldlt": work, "elasticity": work, "details": bench.DETAILS}


def test_line_is_short_and_whole():
    for steps in (5, 20, 500):
        full = _full(steps)
        assert len(json.dumps(full)) > 3 * bench.LINE_BYTES
        text = json.dumps(bench.headline(full))
        assert len(text) <= bench.LINE_BYTES
        line = json.loads(text)
        for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                  "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
            assert line[k] == full[k]
        assert set(line["modes"]) == {"fp64", "fp32", "tf32", "bf16"} and line["roofline"]["kernel"]
        assert line["workload_ms"]["batched_lu"] == {"fp32_refined": 26.3, "fp64": 70.6}


def test_absent_workloads_leave_no_keys():
    full = {k: v for k, v in _full(5).items() if k not in ("batched_lu", "differentiation", "ldlt", "elasticity",
                                                           "cpu_baseline")}
    line = bench.headline(full)
    assert "workload_ms" not in line and "cpu_baseline" not in line
