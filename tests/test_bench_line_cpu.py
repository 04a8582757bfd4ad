"""The benchmark's printed line: the headline fields and the summary, short
enough that the end of a recorded output holds it whole (no GPU)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_printed_line_is_short_and_complete():
    sys.path.insert(0, ROOT)
    import bench

    rnd = 641234.123456789012
    roof = {k: "a note of about forty characters, or more" if k.endswith("source") else rnd for k in
            ("bound", "unit", "kernel", "achieved", "peak", "frac", "peak_source", "peak_measured",
             "frac_of_measured", "peak_measured_source", "executed_flops_per_launch", "model_flops_per_launch",
             "model_over_executed", "traffic", "algorithmic_bytes_per_launch", "dram_gbs_algorithmic",
             "dram_gbs_measured_traffic", "issue_active_pct_ncu", "counts_key", "counts_present")}
    err = {"max": 2.512345678901e-16, "median": 1.3512345678901e-16, "points": 65536, "bound": 1e-12,
           "within_bound": True, "max_spectral": 1.2512345678901e-15, "spectral_points": 4096}
    e2e = {"value": rnd, "unit": "HVP/s", "h2d_bytes_per_step": 1 << 26, "d2h_bytes_per_step": 1 << 25,
           "api": "chessfad_hvp_host (pinned host buffers)", "slices": 0, "ms_per_step": rnd}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 6}
    line = {"metric": bench.METRIC, "value": rnd, "unit": "HVP/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": rnd, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic (seeded PCG64 draws of the workload's distributions)",
            "config": bench.headline_config(65536, 1), "launch": {"evaluation": "structured"}, "dense": roof,
            "roofline": roof, "e2e": e2e, "gpu_launches": 20, "clocks": clocks,
            "fp32_comp": {"value": rnd, "unit": "HVP/s", "dtype": "f32", "ms_per_step": rnd, "e2e": e2e,
                          "roofline": roof, "dense": roof, "error_vs_oracle": err},
            "chunk_sweep": [rnd] * 200, "workloads": {}, "error_vs_oracle": err,
            "cpu_baseline": {"value": rnd, "unit": "HVP/s", "cores": 16, "kind": "oracle", "sample": "x" * 100}}
    for name, kind, how, prec in bench.WORKLOAD_ROWS:
        rate = "hvp_per_s" if kind == "hvp" else "hessians_per_s"
        line["workloads"][f"{name}/{bench.PREC_NAME[prec]}/{kind}/{how}"] = {rate: rnd, "roofline": roof,
                                                                             "error_vs_oracle": err}
    line["summary"] = bench.compact_summary(line)
    short = bench.short_line(line)
    assert len(json.dumps(short)) <= 4096
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert short[key] == line[key], key
    assert short["fp32_comp"]["value"] == rnd and list(short)[-1] == "summary"
    assert len([k for k in short["summary"] if "/" in k]) == len(bench.WORKLOAD_ROWS)
