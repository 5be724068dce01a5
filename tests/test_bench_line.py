"""The line that bench.py prints: every key of the report that its reader needs, unchanged, and short enough to be read
from the end of a run's output."""
import json

import bench

CONTRACT = {"metric": bench.METRIC, "value": 552189256.7, "unit": "elements/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 3.79788, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32 integrate + f64 accumulate", "data": "synthetic " + 60 * "x",
            "config": {"workload": bench.workload_name(128), "variant": "fp32_block", "l2": 50 * "x"},
            "roofline": {"bound": "alu", "frac": 0.45, "kernel": 60 * "x", "peak_source": 80 * "x"},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 7.0e7, "unit": "elements/s", "h2d_bytes_per_step": 51520536,
                    "d2h_bytes_per_step": 4160317536},
            "gpu_launches": 40}
ERROR = {"A_normwise": 9.085342714123159e-08, "A_relative": 0.0035807467599915373, "b_normwise": 9.300396095988013e-08,
         "b_relative": 9.300396095988013e-08, "bar": 1e-05, "within_bar": True, "rows": 93, "entries": 6723}
ROOF = {"bound": "alu", "resource": "fp64", "achieved": 429.53209162777847, "peak": 1059.3873862779533,
        "unit": "GFLOP/s (FP64)", "frac": 0.4054532810107307, "t_roof_ms": 1.539865451609209, "ms": 3.797886276245117}
SCHEDULES = ["fp64_per_type", "fp32_per_type", "fp32_persistent_steal"] + [
    f"fp32_{c}_{s}" for c in ("mlp", "gauss_points") for s in ("queues", "queues_steal", "ordered_steal")]


def _workload(names):
    return {"workload": 150 * "x", "ms": {n: 2.5652480125427246 + k for k, n in enumerate(names)},
            "elements_per_s": {n: 344892967.7263572 for n in names}, "roofline": {n: dict(ROOF) for n in names},
            "error": {n: dict(ERROR) for n in names}, "wall_s": 0.3}


def _report():
    j2 = _workload(SCHEDULES)
    j2["element_loop"] = dict(_workload([n[5:] for n in SCHEDULES[1:]]), error=dict(ERROR))
    batch = {"workload": 150 * "x", "ms": 14.6, "roofline": dict(ROOF), "error": {n: dict(ERROR) for n in "abc"}}
    return dict(CONTRACT, step_roofline=ROOF, error=dict(ERROR, sample=80 * "x"), cpu_baseline={"value": 9226.1},
                variants={n: {"ms_per_step": 3.79788, "zero_ms": 0.42, "step_roofline": dict(ROOF)} for n in bench.VARIANTS},
                errors={n: dict(ERROR) for n in bench.VARIANTS}, first_call_s={n: 0.1 for n in bench.VARIANTS},
                autotuned={n: {"ms": 1.0} for n in bench.VARIANTS}, rows_plan={"blocks": 1},
                spmv={"ms": 1.028, "frac": 0.6471, "fp64_frac": 0.7996, "error": dict(ERROR)},
                neohooke={"deformation": 60 * "x", "fp64_atomic": {"ms": 38.8, "error": dict(ERROR)}},
                workloads={"poisson": _workload(SCHEDULES[:3]), "hybrid": _workload(SCHEDULES), "j2": j2, "batch": batch})


def test_line_is_short_and_keeps_the_contract():
    report = _report()
    line = bench.summary_line(report, "report.json")
    assert len(json.dumps(line)) < 8192 < len(json.dumps(report))
    for key, value in CONTRACT.items():
        assert line[key] == value, key
    assert line["error"] == report["error"] and line["cpu_baseline"] == report["cpu_baseline"]
    assert line["report"] == "report.json" and set(line["variants"]) == set(bench.VARIANTS)
    assert line["workloads"]["hybrid"]["ms"]["fp32_per_type"] == 3.565 and line["workloads"]["batch"]["ms"] == 14.6
    assert line["workloads"]["j2"]["within_bar"] and line["workloads"]["j2"]["element_loop"]["within_bar"]


def test_an_error_past_its_bar_shows():
    report = _report()
    report["workloads"]["hybrid"]["error"]["fp32_mlp_queues"]["within_bar"] = False
    report["errors"]["fp64_rows"]["within_bar"] = False
    line = bench.summary_line(report, "report.json")
    assert not line["workloads"]["hybrid"]["within_bar"] and line["workloads"]["j2"]["within_bar"]
    assert not line["variants"]["fp64_rows"]["within_bar"] and line["variants"]["fp64_atomic"]["within_bar"]


def test_a_run_without_oracle_or_workloads():
    report = {k: v for k, v in _report().items() if k not in ("errors", "workloads", "error", "cpu_baseline")}
    line = bench.summary_line(dict(report, spmv=None, neohooke=None), "report.json")
    assert line["workloads"] == {} and "spmv" not in line and "error" not in line
