"""The line bench.py prints stays short enough to be read whole from the end of a captured output, and
keeps every figure of the headline; the legs' details are left to the record on stderr."""
import json

import bench

LIMIT = 2900  # characters: callers that keep the last 3,000 see all of the line


def record():
    f = 123456.78901234567
    stages = {k: f for k in ("norm", "pair_h", "boys_r", "gemm1", "gemm2", "split", "digest")}
    errors = {f"({a}{b}|{c}g)": {"n": 3, "max_abs_integral": f, "max_abs_err_split": f * 1e-20, "rel_err_fp64": f * 1e-20}
              for a in "ghi" for b in "ghi" for c in "ghi"}
    arm = {"quartets_per_s": f, "ms_per_step": f, "fp64_equiv_tflops": f, "stage_ms_per_step": stages,
           "max_abs_diff_vs_fp64_path": f * 1e-20, "note": "n" * 200}
    leg = dict(arm, workload="w" * 200, oracle_err_per_class=errors)
    return {"metric": bench.METRIC, "value": f, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": f, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": bench.workload_name(4096), "path": "plain FP64",
                                            "l2": "512 MB buffer written between timed steps",
                                            "parallelism": "replicas x1"},
            "fp64_equiv_tflops": f, "integrals_per_s": f * 1e6, "stage_ms_per_step": stages,
            "roofline": {"bound": "compute", "kernel": "axial_main", "unit": "TFLOP/s", "achieved": f, "peak": f,
                         "frac": f, "cublas_dgemm_tflops": f, "traffic": f * 1e6, "peak_source": "p" * 250},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "power_w_max": 1187.44, "samples": 70,
                       "reasons": ["sw_power_cap"]},
            "e2e": {"value": f, "unit": bench.UNIT, "h2d_bytes_per_step": 1015808, "d2h_bytes_per_step": 935886848,
                    "note": "n" * 300},
            "cpu_baseline": {"value": f, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 150},
            "cartesian": dict(leg, fp64_tflops=f), "split": dict(leg, roofline=arm),
            "mixed": {"split": arm, "fp64": arm, "split_max_abs_diff_vs_fp64_on_sample": f, "oracle_err_per_class": errors},
            "split_config": dict(leg, max_abs_err_vs_fp64_path_on_sample=f),
            "routed": {"routed_quartets_per_s": f, "split_only_quartets_per_s": f, "fp64_only_quartets_per_s": f,
                       "routed_max_abs_err_vs_fp64_on_sample": f * 1e-20, "oracle_err_per_class": errors},
            "pairs": {"workload": "w" * 200, "fp64": arm, "split": arm},
            "jk": {"workload": "w" * 200, "fp64": arm, "split": arm}, "sweep": [leg] * 6, "gpu_launches": 140}


def test_line_is_short_and_keeps_the_headline():
    full = record()
    line = bench.headline(full)
    text = json.dumps(line)
    assert len(text) <= LIMIT, len(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches", "fp64_equiv_tflops"):
        assert line[key] == full[key], key
    for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == full["e2e"][key]
    assert line["roofline"]["frac"] == full["roofline"]["frac"]
    assert abs(line["split"]["quartets_per_s"] / full["split"]["quartets_per_s"] - 1) < 1e-5
    assert line["mixed"]["fp64"]["quartets_per_s"] and line["routed"]["routed_quartets_per_s"]


def test_line_of_a_run_with_legs_left_out():
    full = record()
    for leg in bench.LEGS + ("e2e", "cpu_baseline", "sweep"):
        full[leg] = None
    line = bench.headline(full)
    assert line["value"] == full["value"] and line["e2e"] is None and "split" not in line
