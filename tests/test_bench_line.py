"""The benchmark's JSON line (no GPU): short enough for what reads it, with every key of
its contract, whatever the record holds."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

REQUIRED = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
            "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
            "gpu_launches", "clocks")


def _record(bench, long):
    pad = "x" * long
    stages = {s: 0.123456789012345 for s in ("covariance", "cov_finalize", "jacobi", "empty",
                                             "compact", "refine", "sort_sign", "project")}
    forms = {p: {"ms": 2.1003360748291016, "value": 447320.8393930226, "ms_per_step": 1.0,
                 "sweeps": 4, "stage_ms": stages, "errors": {"q": [1e-7] * 20}}
             for p in ("mix", "fp16_mix", "p32", "p64")}
    return {"metric": bench.METRIC, "value": 447320.8393930226, "unit": bench.UNIT, "n_gpus": 1,
            "steps": 20, "warmup": 5, "ms_per_step": 2.1003360748291016, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "precision": "mix"}, "forms": forms,
            "stage_ms_per_step": stages,
            "hbm_kernels": {k: {"frac": 0.5, "how": pad} for k in ("k_syrk_tc", "k_project")},
            "errors": {f"case_{i}": {"eig_rel_err_topk_max": 1.97653980621e-08, "q": [1.0] * 20}
                       for i in range(6)},
            "roofline": {"kernel": "k", "bound": "alu", "achieved": 1.0, "peak": 2.0, "unit": "u",
                         "frac": 0.5, "peak_basis": pad},
            "cpu_baseline": {"value": 86.3, "unit": bench.UNIT, "cores": 16, "kind": "oracle",
                             "sample": pad},
            "oracle_timings": {"how": pad},
            "e2e": {"value": 62146.643771998555, "unit": bench.UNIT, "how": pad,
                    "h2d_bytes_per_step": 1879048192, "d2h_bytes_per_step": 335949312},
            "two_in_flight": {"unit": "u", "a": {"ms_per_fit": 1.6, "value": 2.0}, "how": pad},
            "gpu_launches": 520,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 41},
            "scenes": {"workload": pad, "forms": forms},
            "mixing_100x100x128": {"forms": forms},
            "differentiation": {"workload": pad, "forward_ms": 1.5, "backward_ms": 0.3},
            "batched": {"workload": pad, "forms": forms},
            "paper_shapes_k1": [{"workload": f"shape {i}{pad[:40]}", "mix": {"ms": 1.0}}
                                for i in range(10)]}


def test_line_is_short_and_complete():
    import bench
    for long in (10, 3000):
        rec = _record(bench, long)
        line = bench.summary_line(rec)
        assert len(json.dumps(line)) <= bench.LINE_CHARS
        for key in REQUIRED:
            assert key in line, key
        assert line["value"] == rec["value"] and line["ms_per_step"] == rec["ms_per_step"]
        for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
            assert line["e2e"][key] == rec["e2e"][key]
        assert line["forms_ms"]["mix"] == 2.1


def test_line_of_a_partial_run():
    import bench
    rec = _record(bench, 10)
    for key in ("scenes", "mixing_100x100x128", "differentiation", "batched", "paper_shapes_k1",
                "cpu_baseline", "e2e", "two_in_flight"):
        rec[key] = None
    line = bench.summary_line(rec)
    assert line["value"] == rec["value"] and "e2e" not in line
