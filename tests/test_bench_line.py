"""bench.py's printed line stays whole for a reader that keeps the last 3000
characters of the output; everything measured is in the details (no GPU)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def _line():
    import bench
    roof = {"bound": "fp64", "kernel": "k_flux_update", "achieved": 382.123456789, "peak": 629.28, "unit": "G FP64-pipe lanes/s",
            "frac": 0.6072345678, "hbm_frac": 0.0986300266, "peak_source": "x" * 200, "other": {"a": [1.0] * 200}}
    form = {"value": 158606692.0347288, "edge_iterations_per_s": 1291422945.5719948, "ms_per_step": 15.753181457519531,
            "roofline": roof, "kernels": {"k": {"launches": 1}}}
    err = {"converged_10k": {"cl_rel_err": 7.321592374635663e-06, "cd_rel_err": 1.6188791750116692e-06, "cp_max_abs_err": 2.5661981519972676e-06},
           "bench_cloud_after_timed_steps": {"residual_at_fp64_state": {"rel_l2": 1.5138196063088135e-05}, "cd_rel_err": 8.105696843651378e-08}}
    forms = {"fp64": form, "mixed": dict(form, roofline=dict(roof, kernel="k_flux_update_mixed", avg_launch_ms=0.27969680093, other=dict(roof, kernel="k_qgrad_mixed")), error=err),
             "mixed_speedup_vs_fp64": 5.7066324438397, "batched": dict(form, speedup_vs_sequential=1.7537438594864638, clouds=["c" * 100] * 20),
             "batched_speedup_vs_fp64": 6.173101831685952, "mixed_10m": dict(form, clocks={"sm_mhz": [2070.0] * 500})}
    line = {"metric": bench.METRIC, "value": form["value"], "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": form["ms_per_step"], "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": "naca0012_2p5m", "points": 2498560, "mean_degree": 8.142, "order": 2, "inner_iters": 3, "scheme": "rk4",
                       "mach": 1.2, "aoa_deg": 0.0, "cfl": 0.2, "limiter_K": 1.0, "precision": "fp64", "reorder": "morton",
                       "input_order": "shuffled", "l2": "inputs larger than L2 (working set ~1.7 GB)", "parallelism": "replicas"},
            "edge_iterations_per_s": form["edge_iterations_per_s"], "roofline": roof, "kernels": form["kernels"], "gpu_launches": 360,
            "measured_fma_peaks_gflops": {"fp64_fma_gflops": 1258.1234567}, "e2e": {"value": 123456789.123456, "unit": bench.UNIT,
                                                                                 "h2d_bytes_per_step": 79953920, "d2h_bytes_per_step": 79953928},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 123, "reasons": ["sw_power_cap"]},
            "forms": {k: v for k, v in forms.items() if k != "fp64"}, "tuning": {"flux_variant": 22},
            "cpu_baseline": {"value": 390109.3568258837, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 150}}
    line["summary"] = bench.summary_of(line, forms)
    return line


def test_the_line_is_short_and_complete():
    import bench
    line = _line()
    short, details = bench.split_line(line)
    text = json.dumps(short)
    assert len(text) <= bench.LINE_LIMIT < 3000, len(text)
    back = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "gpu_launches"):
        assert back[k] == line[k], k
    assert back["config"] == line["config"] and back["clocks"] == line["clocks"]
    assert back["e2e"]["h2d_bytes_per_step"] == 79953920 and abs(back["e2e"]["value"] / line["e2e"]["value"] - 1) < 1e-5
    assert set(back["summary"]) == set(line["summary"])
    assert details["details"] is line
