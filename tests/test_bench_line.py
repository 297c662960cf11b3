"""The line that bench.py prints fits what a log reader keeps of a run's output
(4.8 kB), whatever the comparison legs record, and holds the headline's fields as
they were measured."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

X = 12345.678901234567


def _gates():
    dist = {k: X for k in ("min", "p10", "median", "p90", "max")}
    return {"sample": 256, "cost_tol": 1e-6, "one_sided": 0.51953125, "two_sided": 0.02734375, "converged_both": 41,
            "two_sided_converged_both": 0.8780487804878049, "settled_vs_converged": 64, "ratio_minus_1": dist,
            "ratio_minus_1_converged_both": dist, "traj_rel_err": dist, "traj_rel_err_converged_both": dist}


def _leg():
    return {"B": 16384, "ms": X, "raw_solves_per_s": X, "us_per_iteration": X, "mean_iters": X,
            "status_counts": [10298, 139, 5915, 32, 0],
            "roofline": {"bound": "alu", "achieved": X, "peak": X, "unit": "TFLOP/s", "frac": 0.05506117559764456,
                         "algorithmic_flops": 31387150381800.0, "peak_source": "s" * 120, "note": "n" * 150},
            "accuracy": {"reference": "FP64 CPU oracle", "sample": 64, "traj_rel_err_median": X, "gates": _gates()}, "value": X}


def _full():
    rate = {"requests": 5984, "arrivals_s": X, "wall_s": X, "solves_per_s": X, "p50_ms": X, "p99_ms": X, "ok_fraction": 1.0}
    rank = {"candidates": 81920, "selected": 8192, "ms": X, "candidates_per_s": X, "mlp_tflops": X,
            "frac_of_fp32_peak": 0.4019993159594061, "timing": "t" * 110}
    return {
        "metric": "m" * 75, "value": 16616.29787447189, "unit": "solves/s", "n_gpus": 8, "steps": 20, "warmup": 5,
        "ms_per_step": 256.1340698242187, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "precision": "p" * 265, "data": "synthetic (seeded generator)",
        "config": {"workload": "w" * 110, "batch_per_gpu": 8192, "knots_per_gpu": 2050070, "parallelism": "independent instances x8",
                   "l2": "l" * 65, "launch": "k" * 105},
        "raw_solves_per_s": X,
        "within_tol": {"cost_tol": 1e-6, "sample": 256, "fraction": 0.51953125, "rule": "r" * 200, "gates": _gates(),
                       "oracle_self_reproducibility": dict(_gates(), perturbation="x0 * (1 +- 1e-15)")},
        "e2e": {"value": 16567.50165712338, "unit": "solves/s", "h2d_bytes_per_step": 425984, "d2h_bytes_per_step": 236453888,
                "ms_per_step": 256.8884608000076, "api": "a" * 125, "kernels_per_step": 3, "results_equal_device_solve": True},
        "autotune": {"chosen": [8, 32, 1], "calibration": "c", "columns": ["a", "b", "c", "d"], "rows": [[8, 8, 1, 12.34]] * 36},
        "gpu_launches": 40,
        "roofline": {"bound": "alu", "achieved": X, "peak": X, "unit": "TFLOP/s", "frac": 0.06987, "traffic": 361476664832.0,
                     "peak_source": "p" * 230, "frac_of_fp32_peak": 0.06987, "algorithmic_flops_per_launch": X,
                     "fp64_flops_per_launch": 0.0},
        "cpu_baseline": {"value": X, "unit": "solves/s", "cores": 16, "kind": "oracle", "sample": "s" * 85,
                         "single_core": {"value": X, "unit": "solves/s", "cores": 1, "sample": "s" * 50}},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 31},
        "batched_fp64": {"value": X, "raw_solves_per_s": X, "ms_per_step": X, "within_tol": 0.5},
        "plain_fp64_one_instance_per_launch": {"value": X, "raw_solves_per_s": X, "sample": 6, "within_tol": 0.7},
        "levenberg_marquardt": {"raw_solves_per_s": X, "ms_per_step": X, "mean_iters": X, "note": "n" * 300,
                                "within_tol_vs_lm_oracle": 0.5, "gates_vs_lm_oracle": _gates(),
                                "fp64_gpu_on_the_sample": {"gates_vs_lm_oracle": _gates()}},
        "serve": {"workload": "w" * 180, "latency": "l" * 80, "seats_mixed": 106721, "seats_fp64": 89402,
                  "mixed": [dict(rate, rate_per_s=10.0 ** k) for k in (2, 3, 4, 5)],
                  "fp64": [dict(rate, rate_per_s=10.0 ** k) for k in (2, 3, 4, 5)]},
        "other_workloads": {n: {"workload": "w" * 90, "mixed": _leg(), "fp64": _leg(), "vs_stored_oracle": {"mixed": _gates()}}
                            for n in ("pointmass", "arm7", "quad", "dubins")},
        "bic_ranking": {"planar3": rank, "quad": rank},
        "multi_system": {"workload": "w" * 95, "sequential_s": X, "alone_s": {"a": X}, "one_launch_s": X, "graph_note": "n" * 90,
                         "equal_shares": {"graph_s": X}, "work_shares": {"graph_s": X}},
    }


def test_the_printed_line_is_short_and_whole():
    import bench
    full = _full()
    before = json.dumps(full)
    text = json.dumps(bench.compact_line(full))
    assert json.dumps(full) == before          # (--details still gets everything)
    assert "\n" not in text and len(text) <= 4800, len(text)
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "raw_solves_per_s", "e2e", "gpu_launches", "clocks"):
        assert line[k] == full[k], k
    assert line["roofline"]["frac"] == full["roofline"]["frac"]
    assert line["within_tol"]["gates"]["two_sided"] == 0.0273438
    assert line["other_workloads"]["arm7"]["fp64"]["ms"] == 12345.7
    assert line["serve"]["mixed"][3][0] == 1e5 and line["serve"]["columns"][0] == "rate_per_s"


def test_a_run_without_the_comparison_legs():
    import bench
    full = {k: v for k, v in _full().items() if k not in ("levenberg_marquardt", "serve", "other_workloads", "bic_ranking",
                                                          "multi_system", "batched_fp64", "plain_fp64_one_instance_per_launch")}
    line = bench.compact_line(full)
    assert set(line) == set(full) and line["value"] == full["value"]
