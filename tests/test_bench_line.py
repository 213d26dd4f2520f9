"""The benchmark's one line on stdout stays short enough for a reader that keeps
some kilobytes of the output, whatever its legs record (no GPU)."""
import json

import bench


def test_line_is_short():
    args = bench.parse(["--steps", "20", "--warmup", "5"])
    x = 12345678901.123456
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 99,
              "samples_in_timed_region": 99, "samples_total": 999, "period_ms": 10, "timed_region_s": 0.123}
    roofline = {"bound": "alu", "kernel": "k_p2p_refine<fp32x>", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x,
                "traffic": x, "peak_source": "s" * 80, "peak_derived_cross_check": x, "work": "w" * 120,
                "flops_per_test": 12.0, "refine_ms_per_launch": x, "algorithmic_tests_per_launch": x,
                "executed_tests_per_launch": x, "executed_frac": x,
                "hbm": {"algorithmic_bytes_per_join": 10 ** 10, "achieved_gbs": x, "peak_gbs": x, "frac": x,
                        "over": "o" * 40, "peak_source": "p" * 40}}
    leg = {"value": x, "unit": "points/s", "steps": 20, "warmup": 5, "ms_per_step": x, "dtype": "f32+f64",
           "config": {f"key{k}": "v" * 20 for k in range(16)}, "roofline": roofline, "clocks": clocks,
           "fallbacks_per_join": x, "edge_tests_per_s_algorithmic": x, "speedup_vs_fp64_form": x,
           "fp64_form": {"value": x, "roofline": roofline, "clocks": clocks},
           "e2e": {"value": x, "unit": "points/s", "h2d_bytes_per_step": 1 << 33, "d2h_bytes_per_step": 1 << 33,
                   "steps": 20, "api": "a" * 20, "timing": "t" * 60},
           "cpu_baseline": {"value": x, "unit": "points/s", "cores": 16, "kind": "oracle", "sample": "s" * 140,
                            "gpu_vs_oracle": {f"error{k}": x for k in range(8)}}}
    line = bench.one_line(args, "p2p", 1, leg, {f"a_leg_with_a_name_{k}": leg for k in range(7)}, 160)
    assert len(json.dumps(line)) < 4096
    assert {"metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "e2e", "clocks", "gpu_launches"} <= set(line)
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
    assert len(line["legs"]) == 7 and all("value" in v and "e2e" in v for v in line["legs"].values())
