"""The line bench.py prints holds the headline as measured and stays short (no GPU needed)."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def record():
    """A record as run_gpu fills it, with as many rows and as long texts."""
    stages = [{"stage": s, "spin": k, "ms_per_step": 1234.5678, "avg_launch_ms": 1234.5678, "bound": "alu",
               "achieved": 12.34, "unit": "TFLOP/s", "frac": 0.1234} for s in bench.STAGES for k in (0, 2)]
    roof = {"bound": "alu", "achieved": 30.123, "peak": 71.8, "unit": "TFLOP/s", "frac": 0.4321, "traffic": None,
            "kernel": "legendre_synthesis (spin 2, fp32)", "avg_launch_ms": 7.6543, "peak_source": "x" * 100}
    pt = {k: 1.2345678901e10 for k in ("T_synthesis", "T_adjoint", "EB_synthesis", "EB_adjoint")}
    leg = {"value": 1382000000.1, "unit": "lensed points/s", "epsilon": 1e-10, "ms_per_step": 363.456, "steps": 3,
           "per_transform": pt, "arithmetic": "y" * 200, "plan": {"n1": 13122, "W": 13, "sigma": 1.6}, "roofline": roof,
           "stages": stages, "step_roofline": {"t_roof_ms": 10.0, "frac": 0.3}}
    plan = {"ntheta": 4100, "n1": 12288, "n2": 12288, "W": 8, "sigma": 1.4998779296875, "beta": 16.75434}
    mode = {"mode": "restarted FP32 recursion", "restart_every": 64, "restart_bytes": 123456789012, "triples": 12345678901}
    return {
        "metric": "m" * 90, "value": 1382000000.1, "unit": "lensed points/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 36.412, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "d" * 70,
        "data": "s" * 80,
        "config": {"workload": "w" * 120, "lmax": 4096, "nside": 2048, "points": 50331648, "epsilon": 1e-5, "step": "s" * 60,
                   "plan_T": plan, "plan_EB": plan, "l2": "l" * 50,
                   "legendre": {"T": mode, "EB": mode, "plan_creation_s": 0.7}, "parallelism": "single GPU"},
        "per_transform": pt, "roofline": roof, "stages": stages,
        "step_roofline": {"t_roof_ms": 12.345, "t_measured_ms": 36.412, "frac": 0.339, "rule": "r" * 200},
        "measured_peaks": {"fp32_fma_tflops": 71.8, "clocks": {"sm_mhz": 2070}}, "gpu_launches": 400,
        "library": "paper_2304_10431_gb300/libgslens.so",
        "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": ["none"], "samples": 123, "power_w_max": 917.73},
        "e2e": {"value": 1.2e9, "unit": "lensed points/s", "h2d_bytes_per_step": 805453848, "d2h_bytes_per_step": 805453848,
                "ms_per_step": 41.2, "statistic": "median", "ms_mean": 41.3, "api": "a" * 80, "ms_min": 41.0, "ms_max": 42.0,
                "ms_all": [41.23] * 20},
        "tables": leg,
        "tensor_cores": {"what": "t" * 250, "legs": [
            {"maps": m, "tensor_cores": {"call_ms": 100.123}, "cuda_cores": {"call_ms": 200.456}} for m in (32, 64)]},
        "fp64": leg, "lmax5120": {"workload": "z" * 100, "legs": [dict(leg, precision="fp64")] * 4},
        "cpu_baseline": {"value": 19.3, "unit": "lensed points/s", "cores": 16, "kind": "oracle", "sample": "q" * 150,
                         "seconds_per_step": 6.6},
    }


def test_line_is_short_and_keeps_the_headline():
    full = record()
    text = json.dumps(bench.compact(full))
    assert len(text) <= 4096 < len(json.dumps(full))
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "gpu_launches", "library", "clocks"):
        assert line[k] == full[k]
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == full["e2e"][k]
    for k in ("workload", "lmax", "nside", "points", "epsilon", "step", "l2", "parallelism"):
        assert line["config"][k] == full["config"][k]
    assert line["roofline"]["frac"] == full["roofline"]["frac"] and line["fp64"]["ms_per_step"] == 363.456


def test_line_without_the_other_legs():
    full = record()
    for k in ("tables", "tensor_cores", "lmax5120"):
        full[k] = None
    del full["cpu_baseline"]
    full["e2e"] = full["fp64"] = None
    full["recursion"] = {"unavailable": "no memory"}
    line = bench.compact(full)
    assert line["e2e"] is None and line["cpu_baseline"] is None and line["recursion"] == {"unavailable": "no memory"}
