"""The line that bench.py prints holds every key of its contract and is short enough to be
kept whole by a reader of the last 3,000 characters."""
import json

import bench


def full_line():
    text = "x" * 160
    forms = {"unit": "DOF-stage/s", "batched": {"value": 3.14458288620e11, "loop_value": 1.0, "workload": text},
             "implicit_backward_euler": {"block_jacobi": {"value": 8.26e8}, "workload": text}}
    for key, wname, prec, red in bench.FORMS:
        forms[key] = {"value": 1.4700312364137e11, "workload": text, "tile": {"grid": 456}, "error": {"copy": text}}
    desc = max((w["desc"] for w in bench.WORKLOADS.values()), key=len)
    return {"metric": "DOF-stage updates/s", "value": 2.518697327886e11, "unit": "DOF-stage/s", "n_gpus": 1, "steps": 2000,
            "warmup": 50, "ms_per_step": 0.62447519302368, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": desc, "name": "n" * 48, "K": 8192, "Np": 15, "Q": 256, "dof": 31457280,
                       "reduction": "default", "tile": {"elems_per_cta": 1, "threads_per_cta": 160, "pipeline_stages": 3,
                                                        "grid": 456, "tensor_cores": 0},
                       "l2": "inputs larger than L2 (state x2 + residual = 377 MB), no flush", "parallelism": "replicas x1"},
            "repeats": {"n": 5, "ms_per_step_median": 1.593017578125, "ms_per_step_min": 1.5924495697021483,
                        "ms_per_step_max": 1.5944031715393066, "spread_pct": 0.1226352969348659},
            "roofline": {"bound": "hbm", "achieved": 5396.032845891043, "peak": 6786.2, "unit": "GB/s",
                         "frac": 0.7951479245956563, "peak_source": "measured", "traffic": 421379800.0,
                         "algorithmic_bytes_per_dof_step": 76, "algorithmic_bytes_per_launch": 478150656.0,
                         "kernel": "stage_kernel_ws (5 launches per step; average over the mix)"},
            "error": {"l2_rho": 4.486670862738493e-08, "l2_u_over_U": 1.5858788743930517e-07,
                      "max_abs_u_over_U": 4.655748073717577e-07, "max_abs_rho": 1.816357551032155e-07, "copy": text},
            "cpu_baseline": {"value": 33840415.21419811, "unit": "DOF-stage/s", "cores": 1, "kind": "oracle",
                             "sample": text, "all_cores": {"value": 1.0, "sample": text}},
            "e2e": {"value": 127383648907.14204, "unit": "DOF-stage/s", "steps": 20, "h2d_bytes_per_step": 251658240,
                    "d2h_bytes_per_step": 2949120, "input_dtype": "f32", "path": text,
                    "serial": {"value": 1.0, "path": text}},
            "gpu_launches": 10000, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 3,
                                              "power_w_median": 400.06}, "mass_after": 1.0, "forms": forms}


def test_line_is_whole_in_the_last_3000_characters():
    full = full_line()
    line = bench.contract_line(full)
    assert len(json.dumps(line)) < 2700 < len(json.dumps(full))
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in line
    for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == full["e2e"][key]
    assert set(line["forms"]) == {k for k, *_ in bench.FORMS} | {"batched"}
    assert full["forms"] and "path" in full["e2e"]  # the full line is left as it is
    assert json.loads(json.dumps(line)) == line
    assert bench.contract_line(dict(full, forms=None, error=None, cpu_baseline=None))["error"] is None
