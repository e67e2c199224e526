"""The benchmark's last line: one short JSON line that a log's end keeps whole,
with the metric, the end-to-end figure and the clocks; the details stand before it."""
import json

import bench


def _full():
    pi = 3.141592653589793 * 1e3
    long = "w" * 600
    return {"metric": bench.METRIC, "value": pi, "unit": "solves/s", "n_gpus": 8, "steps": 1000, "warmup": 100,
            "ms_per_step": pi, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f16/f32/f64",
            "data": "synthetic (the paper's H-equation, x0=ones)",
            "config": {"workload": bench.WORKLOAD, "N": 4096, "c": list(bench.SWEEP), "mode": "GMRESIR16",
                       "l2": "flushed between steps (256 MiB write)", "parallelism": "replicas x8", "concurrency": long,
                       "cuda_device_max_connections": 32},
            "roofline": {"bound": "tensor", "achieved": pi, "peak": pi, "unit": "TFLOP/s", "frac": pi, "traffic": 171520000,
                         "kernel": "k_gemv_residual", "launches": 9999, "avg_us": pi, "work_per_launch": pi * 1e9,
                         "peak_kind": long},
            "roofline_lu": {"note": long}, "kernels": {f"k{i}": {"total_ms": pi, "peak_kind": long} for i in range(8)},
            "e2e": {"value": pi, "unit": "solves/s", "h2d_bytes_per_step": 163840, "d2h_bytes_per_step": 163840,
                    "path": long},
            "gpu_launches": 123456,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0,
                       "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_power_cap", "sw_thermal_slowdown"], "samples": 9},
            "per_c": {str(c): {"ms": pi, "note": long} for c in bench.SWEEP}, "speedup_vs_fp64lu": pi,
            "batched": {"solves_per_s": pi, "workload": long}, "large": {"ms_to_solution": pi, "workload": long},
            "serving": {"p50_ms": pi, "p99_ms": pi, "workload": long}, "serving_fp64lu": {"p50_ms": pi, "note": long},
            "cpu_baseline": {"value": pi, "unit": "solves/s", "cores": 144, "kind": "oracle", "sample": long}}


def test_last_line_is_short_and_complete():
    full = _full()
    lines = bench.report(full)
    assert len(lines[-1]) <= bench.LINE_LIMIT and "\n" not in lines[-1], len(lines[-1])
    short = json.loads(lines[-1])
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
              "gpu_launches"):
        assert short[k] == full[k], k
    assert abs(short["value"] / full["value"] - 1) < 1e-6 and abs(short["ms_per_step"] / full["ms_per_step"] - 1) < 1e-6
    assert {"workload", "parallelism", "l2"} <= set(short["config"])
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(short["e2e"])
    assert short["clocks"]["reasons"] == full["clocks"]["reasons"] and short["clocks"]["sm_mhz"] == 2070.0


def test_details_stand_before_the_line_and_are_no_json_lines():
    full = _full()
    details = bench.report(full)[:-1]
    seen = {}
    for text in details:
        mark, key, body = text.split(" ", 2)
        assert mark == "#" and "\n" not in text
        seen[key] = json.loads(body)
    assert seen == {k: v for k, v in full.items() if isinstance(v, dict)}


def test_workloads_left_out_leave_their_summaries_out():
    full = _full()
    for k in ("batched", "large", "serving", "serving_fp64lu", "cpu_baseline", "speedup_vs_fp64lu"):
        del full[k]
    short = json.loads(bench.report(full)[-1])
    assert short["also"] == {} and "cpu_baseline" not in short
