"""The benchmark's printed line: short enough to be read whole from the end of
a run's output, with everything that qualifies the headline in it (no GPU)."""
import argparse
import json


def _full():
    """A record as large as a default run's: eight levels, five arms, three legs."""
    import bench

    args = argparse.Namespace(grid=128, gamma=0.1, tol=1e-8, lump="diag", krylov="cg")
    x = 1.0 / 3.0
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["hw_slowdown", "sw_power_cap"], "samples": 123}
    arm = {"time_to_tol_ms": 123.456, "iterations": 28, "nnz_per_level": [14581760] * 8, "final_relres": x,
           "eager_breakdown_ms": {k: x for k in ("total", "vcycle_kernels", "pcg_kernels", "other_host_and_checks")}}
    c3 = {f"gamma{g}_{p}": arm for g in (0.0, 0.1) for p in ("fp64", "fp32", "fp32_bf16")}
    c4 = {k: {"ms": 123.456, "solves_per_s": 51.98, "iterations_max": 38}
          for k in ("fp64_single", "fp32_k1", "fp32_k8", "fp32_k32", "fp32_k64")}
    c5 = {"requests": 2400, "failed": 0, "solves_per_s": 198.12, "p50_ms": 98.123, "p99_ms": 258.123, "max_ms": x}
    return {
        "metric": bench.METRIC, "value": 48.5 + x, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 20.6 + x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": bench.workload_config(args), "iterations": 28,
        "levels": [{"n": 2097152, "nnz_galerkin": 14581760, "spmv": "sell32", "bytes_per_cycle": x}] * 8,
        "roofline": {"kernel": "relax_pre_residual level 0", "bound": "hbm", "achieved": x * 1e4, "peak": 6778.7,
                     "unit": "GB/s", "frac": x, "traffic": x * 1e9, "peak_source": "measured (file)",
                     "algorithmic_bytes_per_launch": x * 1e9, "avg_launch_ms": x, "launches": 140,
                     "fp64": {"frac": x, "peak_source": "derived"}},
        "vcycle_GBps": x * 1e4, "top_kernels": [{"kernel": "relax_post L0", "ms": x}] * 12,
        "setup_phases_ms": {f"phase_{i}_by_level": [x] * 8 for i in range(8)}, "setup_roofline": {"levels": [x] * 8},
        "solve_ms_per_level": {f"L{i}": x for i in range(8)},
        "e2e": {"value": 45.0 + x, "unit": bench.UNIT, "h2d_bytes_per_step": 200000000, "d2h_bytes_per_step": 16777216,
                "steps": 5},
        "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 200,
                         "phases_s": {"setup": x}},
        "arms": {k: arm for k in ("galerkin", "gamma_0.01", "gamma_0.1", "gamma_1.0", "adaptive_from_1.0")},
        "communication": {"parts": [arm] * 4},
        "legs": {"c3_precision_27pt_192": {"arms": c3, "clocks": clocks, "wall_s": 9.0},
                 "c4_batched_lognormal_160": {"arms": c4, "clocks": clocks, "wall_s": 9.0},
                 "c5_serving": dict(c5, clocks=clocks, wall_s=14.0)},
        "clocks": clocks, "gpu_launches": 123456,
    }


def test_line_is_short_and_complete():
    import bench

    full = _full()
    text = json.dumps(bench.headline(full))
    assert "\n" not in text and len(text) < 2800, len(text)
    line = json.loads(text)
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype",
              "data", "config", "iterations", "clocks", "gpu_launches"):
        assert line[k] == full[k], k
    for k in ("value", "ms_per_step", "vcycle_GBps"):
        assert abs(line[k] - full[k]) <= 5e-6 * full[k], k
    assert line["e2e"]["h2d_bytes_per_step"] == 200000000 and line["e2e"]["d2h_bytes_per_step"] == 16777216
    assert line["roofline"]["traffic"] > 0 and line["cpu_baseline"]["cores"] == 16
    assert line["arms_ms"]["adaptive_from_1.0"] == 123.456
    assert line["legs"]["c4_batched_lognormal_160"]["fp32_k64"] == 123.456
    assert line["legs"]["c5_serving"]["p99_ms"] == 258.123


def test_line_without_the_optional_parts():
    import bench

    full = dict(_full(), e2e=None, cpu_baseline=None, arms=None, legs=None, clocks=None, vcycle_GBps=None)
    full["roofline"] = {k: v for k, v in full["roofline"].items() if k != "fp64"}
    line = bench.headline(full)
    assert line["e2e"] is None and line["arms_ms"] is None and line["legs"] is None and line["clocks"] is None
    full = dict(_full(), legs={"c5_serving": {"error": "RuntimeError: " + "x" * 500, "wall_s": 1.0}})
    assert len(bench.headline(full)["legs"]["c5_serving"]["error"]) <= 80
