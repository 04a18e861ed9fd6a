"""The benchmark's printed line: short enough to be kept whole by what records a run's output (the full result of a
default run is 26 000 characters), with every figure of the timed step."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _full(n_studies):
    x = 12.345678901234567

    def arm():
        return {"seconds_median": x, "seconds": [x] * 8, "updates": [11] * 8, "log_evidence": [x] * 8,
                "breakdown_ms": {"solves_per_level": [x] * 5, "wall_ms": x}}
    run = {f"study_of_a_long_descriptive_name_{i}": {"workload": "w", "plain": arm(), "surrogate": arm(),
                                                     "speedup_surrogate_vs_plain": x, "speedup_ci95": [x, x]}
           for i in range(n_studies)}
    run["smc_fp64_h16"] = {"seconds_median": x, "roofline": {"frac": x}}
    levels = {str(N): {"evals_per_s": x * 1e6, "update_ms": x, "evals": 24000, "solve_launch_ms": x,
                       "solve_evals_per_s": x * 1e6, "solve_kernel": "k", "smem_frac": x} for N in (8, 16, 32, 64)}
    roof = {"kernel": "k", "bound": "alu", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "peak_source": "p" * 90}
    return {"metric": "likelihood evals/s per mesh level", "value": x * 1e6, "unit": "evals/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32+df64", "data": "synthetic", "config": {"workload": "w", "step": "s" * 300, "l2": "flushed"},
            "per_level": levels, "roofline": roof, "roofline_smem": roof,
            "e2e": {"value": x * 1e6, "unit": "evals/s", "h2d_bytes_per_step": 1024000, "d2h_bytes_per_step": 1056000},
            "gpu_launches": 5940, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 9},
            "seconds_to_posterior": run, "batched_uneven": {"speedup": x, "differing": [{"problem": 1}] * 50},
            "cpu_baseline": {"value": x, "unit": "evals/s", "cores": 16, "kind": "oracle", "sample": "s" * 200}}


def test_headline_is_short_and_complete():
    import bench
    for n in (0, 8, 60):
        full = _full(n)
        assert n == 0 or len(json.dumps(full)) > bench.LINE_CHARS
        line = json.loads(json.dumps(bench.headline(full)))
        assert len(json.dumps(line)) <= bench.LINE_CHARS
        for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
                  "config", "gpu_launches", "clocks"):
            assert line[k] == full[k]
        for a, b in ((line["value"], full["value"]), (line["ms_per_step"], full["ms_per_step"]),
                     (line["e2e"]["value"], full["e2e"]["value"]),
                     (line["per_level"]["64"]["evals_per_s"], full["per_level"]["64"]["evals_per_s"])):
            assert abs(a / b - 1) < 1e-6
        assert set(line["e2e"]) == set(full["e2e"]) and line["cpu_baseline"]["cores"] == 16
    assert bench.headline(_full(0))["studies"]["smc_fp64_h16"] == {"s": [12.35]}
