"""The printed line of bench.py is short enough to be read back from the end of a
log (under 2,500 characters) whatever the full record holds, and keeps the keys
of the benchmark contract."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

CLASS = {"launches": 13957, "avg_us": 11.53, "share": 0.0463, "achieved_GBs": 1289.5, "frac_of_hbm": 0.19,
         "mb_per_launch": 14.87, "residency": "l2-resident"}
FORM = {"value": 43.03024082542423, "ms_per_step": 116.19735107421874, "hessian_applies_per_step": 5.0,
        "outer_iters": 4, "final_relres": 1.5372564634948092e-09, "setup_s": 0.03503775999999448,
        "kernel_classes": {f"class_{k}": CLASS for k in range(16)}, "levels": {"state": [784385, 107500, 9585, 847]}}
RUN = {"time_to_1e-8_s": 2.076456256, "hessian_matvecs_per_s": 523.9696222138955, "setup_s": 0.0961,
       "kernels": {f"class_{k}": CLASS for k in range(16)}}


def record():
    return {
        "metric": bench.METRIC, "value": 43.03024082542423, "unit": bench.UNIT, "n_gpus": 8, "steps": 20, "warmup": 5,
        "ms_per_step": 116.19735107421874, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32+f64", "data": "synthetic", "config": {"workload": "lshape1025_checkerboard", "note": "x" * 480},
        "time_to_1e-8_s": 0.11619735107421875, "gpu_launches": 66975,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 300},
        "roofline": {"bound": "hbm", "achieved": 3361.4, "peak": 6781.8, "unit": "GB/s", "frac": 0.4957,
                     "traffic": 51123456.0, "peak_source": "measured", "launches": 1116,
                     "avg_us": 15.39, "kernel": "z" * 200},
        "kernels": {f"class_{k}": CLASS for k in range(16)},
        "solve_phase": {"alg_bytes": 2.0e11, "solve_s": 0.0746766, "achieved_GBs": 2749.2, "frac": 0.4054},
        "e2e": {"value": 43.14684498308243, "unit": bench.UNIT, "h2d_bytes_per_step": 51169305,
                "d2h_bytes_per_step": 12582928, "ms_per_step": 115.88332824707031, "timing": "t" * 100},
        "forms": {f: FORM for f in ("mixed", "fp64", "refine")},
        "batch": dict({f: RUN for f in ("mixed", "mixed_block", "mixed_autotuned", "fp64", "fp64_block",
                                        "fp64_autotuned")}, workload="16 squares"),
        "cube": dict({f: RUN for f in ("mixed", "fp64", "mixed_matrix_free")}, m=16581375),
        "dense_fp64": {"dfma_tflops": 1.058, "spd_inverse": {"n": 847, "ms": 1.567, "tflops": 0.388, "note": "n"}},
        "cpu_baseline": {"value": 2.72, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "host": {"nproc": 16}},
        "speedup_mixed_vs_fp64": 1.7776550189113494, "speedup_refine_vs_fp64": 1.1529023607783797}


def test_line_is_short_and_complete():
    full = record()
    line = bench.headline(full, "bench_detail.json")
    text = json.dumps(line)
    assert len(json.dumps(full)) > 10000 and len(text) < 2500 and "\n" not in text, len(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches"):
        assert line[k] == full[k], k
    assert line["clocks"] == {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"]}
    assert {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")} == {
        k: full["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert line["forms"]["mixed"]["ms_per_step"] == 116.1974 and line["detail"] == "bench_detail.json"


def test_whole_solves_are_not_labelled_as_hbm_traffic():
    t = bench.kernel_table({"cg_one_launch": {"launches": 2, "ms": 0.4, "bytes": 4.8e8},
                            "cg_spmv_l0": {"launches": 2, "ms": 0.04, "bytes": 1.4e8}})
    assert t["cg_one_launch"]["residency"].startswith("cached") and t["cg_spmv_l0"]["residency"] == "hbm"


def test_parts_that_were_not_run_are_left_out():
    full = record()
    full["batch"]["mixed"] = {"status": -5}  # a part that failed has no rate
    assert "mixed" not in bench.headline(full, "d.json")["batch"]
    for k in ("batch", "cube", "dense_fp64", "cpu_baseline"):
        del full[k]
    full["roofline"] = full["solve_phase"] = full["e2e"] = None
    line = bench.headline(full, "d.json")
    assert not {"batch", "cube", "dense_fp64", "cpu_baseline"} & set(line)
