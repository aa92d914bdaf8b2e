"""The line that bench.py prints: short enough that the end of a log holds it
whole, with the keys of its contract, whatever sections were measured."""
import json

import bench


def _solve(extra):
    return {"kappa": 0.13712345678, "solver": "bicgstab", "wall_s": 0.0213193921999952, "iters": 210,
            "reliable_updates": 4, "status": 0, "true_residual": 5.32386385844e-11, "dslash_calls": 1234.0,
            "phase_s": {k: 0.00123456789 for k in "abcd"}, "all_wall_s": [0.021319392199995] * 3, **extra}


def test_line_is_short_and_complete():
    roof = {"bound": "hbm", "achieved": 6478.245418048674, "peak": 6793.1, "unit": "GB/s", "frac": 0.9581927580719,
            "traffic": 595310336.0, "peak_kind": "measured copy bandwidth (burst)", "bytes_per_site": 576,
            "frac_of_nominal_8tbs": 0.8097806772560843}
    num = 12345.678901234567
    names = ["f16", "f32", "f64", "f16_gauge_fixed", "k130_f64", "k130_f16", "k130_f16_bicgstab", "k130_f32_bicgstab",
             "k130_f16_bicgstab_gauge_fixed"]
    batched = {i: {"wall_s": 0.123456789, "speedup_vs_sequential_same_inner": 1.23456789,
                   "speedup_vs_plain_f64": 12.3456789, "persistent_launch_wall_s": 0.123456789} for i in ("f32", "f16")}
    line = {
        "metric": bench.METRIC, "value": num, "unit": "Gflops", "n_gpus": 1, "steps": 1000, "warmup": 20,
        "ms_per_step": 0.0897654321012345, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": bench.DATA, "config": bench.headline_config(bench.DIMS, 1), "dslash_gbs": num,
        "roofline": roof, "mhat": {"ms_per_step": num, "value": num, "unit": "Gflops", "steps": 500, "note": "x" * 90},
        "graph": {"ms_per_step": num, "value": num, "unit": "Gflops", "note": "x" * 60}, "gpu_launches": 12345,
        "paper_context": {"note": "x" * 200},
        "variants": {n: {"value": num, "frac": 0.912345678, "ms_per_step": 0.0456789012, "note": "x" * 200, **roof}
                     for n in ("f16", "f64", "f32_tg", "f16_tg", "f16_staged")},
        "e2e": {"value": num, "unit": "Gflops", "steps": 50, "h2d_bytes_per_step": 100663296,
                "d2h_bytes_per_step": 100663296, "overlap": "x" * 130},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 400, "reasons": ["sw_power_cap"]},
        "solve": {**{n: _solve({"speedup_vs_f64": 6.681818181}) for n in names}, "config": {"note": "x" * 300}},
        "batch": {"point": {"batched": batched}, "mixed": {"batched": batched}, "tune": "x" * 3000,
                  "mrhs_dslash": {"us_per_launch": 236.123456, "gbs": 3812.123456}},
        "learned_preconditioner": {
            "training": {"loss_first": 0.123456789, "loss_last": 0.0123456789, "wall_s": 12.3456789},
            **{d: {n: _solve({}) for n in ("fcg_trained", "fcg_series", "cgnr_plain", "cg_plain_f64", "cg_mixed_f16")}
               for d in ("16x16x16x32", "32x32x32x64")}, "config": {"note": "x" * 500}},
        "cpu_baseline": {"value": 19.27163922738449, "unit": "Gflops", "cores": 16, "kind": "oracle", "sample": "x" * 90,
                         "single_thread_gflops": 1.074345541249023,
                         "oracle_cg_24x24x24x48": {"wall_s": 98.61292329, "iterations": 446, "note": "x" * 300}},
    }
    out = bench.headline_line(line)
    text = json.dumps(out)
    assert len(text) < 3000, len(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline"):
        assert k in out, k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert out["e2e"][k] == line["e2e"][k]
    assert out["value"] == num and out["ms_per_step"] == line["ms_per_step"]
    # the same without the long sections (--quick, --no-solve, --no-cpu)
    for k in ("solve", "batch", "learned_preconditioner", "cpu_baseline"):
        del line[k]
    assert len(json.dumps(bench.headline_line(line))) < 3000
