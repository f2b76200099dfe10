"""The line that bench.py prints stays short enough to be read back from the end
of a program's output, and keeps what it is read for."""
import json

import bench


def record():
    roof = {"bound": "alu", "achieved": 4.1247, "peak": 1.25, "unit": "TFLOP/s", "frac": 3.2998,
            "dfma_loop_tflops": 1.0558, "frac_of_dfma_loop": 3.9067, "traffic": None,
            "kernel": "k_xsweep_2d_f64 + k_ysweep_2d_f64 <euler,fp64>",
            "kernel_share_of_step": 0.9547, "flops_per_point_stage": 1623.4,
            "peak_source": "x" * 80, "hbm_achieved_gbs": 345.5}
    form = {"value": 803.389, "ms_per_step": 3.1574, "note": "x" * 70}
    sub = {"value": 2151.49, "ms_per_step": 12.7473, "roofline": roof, "clocks": {"samples": 6},
           "graph": form, "workload": "x" * 150, "timing": "x" * 100}
    return {"metric": bench.METRIC, "value": 804.778, "unit": "Mpoint-updates/s", "n_gpus": 1,
            "steps": 20, "warmup": 5, "ms_per_step": 3.175, "higher_is_better": True,
            "us_per_step": 3175.04, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "no_graph": form, "persistent": dict(form, graph_replay=form),
            "config": {"workload": "x" * 120, "instances": 2048, "points": 2555200,
                       "precision": "fp64", "l2": "x" * 45, "timing": "x" * 60, "tile_variant": 2,
                       "size_classes": {"stage1_ms": [[0.1] * 5] * 5},
                       "autotune_stage1_ms": [1.1921] * 5, "parallelism": "x" * 36},
            "roofline": roof,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 30},
            "gpu_launches": 100, "point_updates_timed": 51104000.0,
            "fp32": {"value": 6794.617, "ms_per_step": 0.3761, "roofline": roof, "persistent": form},
            "e2e": {"value": 676.368, "unit": "Mpoint-updates/s", "h2d_bytes_per_step": 122665984,
                    "d2h_bytes_per_step": 122665984, "steps": 10},
            "cpu_baseline": {"value": 13.55115, "unit": "Mpoint-updates/s", "cores": 16,
                             "kind": "oracle", "single_thread": 0.85126, "sample": "x" * 200},
            "configs": {**{k: {p: sub for p in precs} for k, _, precs, _, _ in bench.OTHER_CONFIGS},
                        "euler2d_adjoint_512": sub, "burgers_adjoint_256x800": sub},
            "gpu_launches_configs": 1361}


def test_headline_is_short_and_complete():
    d = record()
    line = json.dumps(bench.headline(d), separators=(",", ":"))
    assert len(line) <= 2900 and len(json.dumps(d)) > 10000
    got = json.loads(line)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "clocks",
              "gpu_launches", "e2e"):
        assert got[k] == d[k]
    assert got["config"]["workload"] == d["config"]["workload"] and got["cpu_baseline"]["value"] > 0
    assert got["roofline"]["frac"] == 3.2998 and got["fp32"]["value"] == 6794.617
    assert got["configs"].keys() == d["configs"].keys()
    assert got["configs"]["burgers1d_n400"]["fp64"] == {"value": 2151.49, "roofline": {"frac": 3.2998}}


def test_a_failed_workload_shows_its_error():
    d = record()
    d["configs"]["burgers1d_n400"]["fp64"] = {"error": "RuntimeError()"}
    d["configs"]["euler2d_adjoint_512"] = {"error": "RuntimeError()"}
    c = bench.headline(d)["configs"]
    assert c["burgers1d_n400"]["fp64"] == {"error": "RuntimeError()"} == c["euler2d_adjoint_512"]
