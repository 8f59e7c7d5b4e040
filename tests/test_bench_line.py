"""The one line that the benchmark prints: short enough that a reader who keeps
the last 3,000 characters of the output has all of it, and complete in the keys
that a reader of the figures needs."""
import json

import pytest

import bench

LONG = 12345.678901234567
KERNELS = ["level0_step", "level0_residual_restriction", "outer_Ap", "level0_first_step",
           "level0_prolongation"]
PRECISIONS = ["fp64", "mixed32", "mixed16"]
WORKLOADS = ["poisson2d_sipg_p1_tri_32x32", "convdiff2d_ldg_upwind_q2_512x512_pe1",
             "convdiff2d_ldg_upwind_q2_512x512_pe100", "convdiff2d_ldg_upwind_q2_512x512_pe10000",
             "poisson3d_sipg_p2_tet_48cubed"]


def record(steps):
    """A full record as the default run makes it, every number at full length."""
    roof = {"bound": "hbm", "achieved": LONG, "peak": LONG, "unit": "GB/s", "frac": LONG,
            "peak_kind": "measured hbm_gbs", "bytes_per_iteration": 1234567890,
            "ms_per_iteration": LONG, "bytes_by_part": {f"part{k}": LONG for k in range(20)}}
    open_loop = {"rate_per_s": LONG, "solves_per_s": LONG, "p50_ms": LONG, "p99_ms": LONG,
                 "per_mesh_p50_ms": {w: LONG for w in WORKLOADS}}
    serving = {"saturated": {"solves_per_s": LONG, "wall_s": LONG, "p50_ms": LONG, "p99_ms": LONG},
               "open_loop_0.5x": open_loop, "open_loop_1.5x": open_loop,
               "per_mesh": {w: open_loop for w in WORKLOADS}}
    return {
        "metric": bench.METRIC, "value": LONG, "unit": "solves/s", "n_gpus": 1, "steps": steps,
        "warmup": 3, "ms_per_step": LONG, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": bench.WORKLOAD, "dofs": 1310720, "elements": 131072, "block": 10,
                   "nnzb": 523264, "levels": 9, "candidates": 4, "tol": 1e-10,
                   "solver": "CG (flexible for mixed)",
                   "cycle": {"dense_first_level": 4, "dense_n": 2048, "folded": 1},
                   "l2": "inputs larger than L2 (A 419 MB FP64 / 209 MB FP32 per pass), no flush",
                   "parallelism": "replicas x1"},
        "iterations": {"mixed": [3348] * steps, "fp64": [3348] * steps},
        "rel_residual": {"mixed": LONG, "fp64": LONG, "e2e_host_check": LONG},
        "fp64": {"value": LONG, "unit": "solves/s", "ms_per_step": LONG, "p50_ms": LONG, "p99_ms": LONG},
        "mixed16": {"value": LONG, "unit": "solves/s", "ms_per_step": LONG,
                    "iterations": [3348] * steps, "rel_residual": LONG, "storage": "x" * 80},
        "p50_ms": LONG, "p99_ms": LONG, "setup_s": LONG, "generate_s": LONG,
        "roofline": dict(roof, kernel="k" * 100, traffic=LONG, launches=12345, avg_launch_us=LONG),
        "roofline_iteration": {p: roof for p in PRECISIONS},
        "level0_kernels": {k: {"avg_us": LONG, "frac": LONG, "launches": 10000} for k in KERNELS},
        "error_vs_oracle": dict({p: LONG for p in PRECISIONS}, what="w" * 120),
        "e2e": {"value": LONG, "unit": "solves/s", "h2d_bytes_per_step": 10485760,
                "d2h_bytes_per_step": 10485760},
        "gpu_launches": 130580000,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 100, "samples_under_load": 100,
                   "reasons": ["sw_power_cap", "hw_thermal_slowdown"]},
        "oracle": {p: {"iterations": 3348, "rel_residual": LONG} for p in PRECISIONS},
        "cpu_baseline": {"value": LONG, "unit": "solves/s", "cores": 1, "kind": "oracle", "sample": "s" * 260},
        "serving": {"mixed": serving, "fp64": serving, "peak_bytes": 123456789, "requests": 128},
        "other_workloads": [{"workload": w, "level_dofs": list(range(100000, 100009)),
                             "precisions": {p: {"solves_per_s": LONG, "iterations": 12345,
                                                "roofline_iteration": roof} for p in PRECISIONS}}
                            for w in WORKLOADS],
        "other_workloads_clocks": {"sm_mhz": 2070.0},
    }


@pytest.mark.parametrize("steps", [1, 20])
def test_line_is_short_and_complete(steps):
    rec = record(steps)
    text = json.dumps(bench.compact_line(rec))
    assert len(text) <= 2900
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
                "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
                "gpu_launches", "clocks", "roofline", "cpu_baseline", "p50_ms", "p99_ms"):
        assert key in line
    assert line["config"] == rec["config"] and line["gpu_launches"] == rec["gpu_launches"]
    assert line["e2e"]["h2d_bytes_per_step"] == rec["e2e"]["h2d_bytes_per_step"]
    assert line["iterations"] == {"mixed": [3348], "fp64": [3348]}
    assert abs(line["value"] / rec["value"] - 1) < 1e-5
    assert set(line["serving"]) == {"mixed", "fp64"} and len(line["other_workloads"]) == 5


def test_line_of_a_run_without_the_optional_parts():
    rec = record(3)
    for key in ("serving", "other_workloads", "other_workloads_clocks", "cpu_baseline", "oracle"):
        del rec[key]
    rec["error_vs_oracle"] = None
    rec["roofline"].update(achieved=None, frac=None, traffic=None)
    line = json.loads(json.dumps(bench.compact_line(rec)))
    assert line["roofline"]["frac"] is None and "serving" not in line and "error_vs_oracle" not in line
