"""bench.py's line on stdout (CPU only): the measurement's own keys whole, the other
workloads' headline figures, and short enough to be read back from a log's end;
the traversal's bound by the DRAM bytes measured on its source."""
import json
import os
import sys

import pytest


@pytest.fixture(scope="module")
def bench():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    if root not in sys.path:
        sys.path.insert(0, root)
    argv, sys.argv = sys.argv, ["bench.py"]
    try:
        import bench as b
    finally:
        sys.argv = argv
    return b


def full_line(bench, extra=0):
    load = {"load": 0.8, "batches_per_s": 1 / 3}
    arms = {f"arm{k}": {"p50_ms": 1 / 3, "p99_ms": 2 / 3, "mean_ms": 0.5, "queries_per_s": 1e9 / 3} for k in range(3)}
    stream = {"workload": "w" * 300, "loads": [dict(load, **arms) for _ in range(3)],
              "capacity_queries_per_s": {f"arm{k}": 1e9 / 3 for k in range(6)}, "tuned": {"x": [1 / 3] * 100}}
    err = {"subset": "s" * 200, "results": {"fp32": {"rel_err_max": 1e-6}, "fp16": {"rel_err_max": 2e-6}}}
    return {"metric": bench.METRIC, "value": 12345678.901234567, "unit": "queries/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 329.123456789, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": bench.workload_config(8192, 1 << 22, 1),
            "e2e": {"value": 1e7 / 3, "unit": "queries/s", "h2d_bytes_per_step": 671088640, "d2h_bytes_per_step": 16777216},
            "gpu_launches": 280, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "roofline": {"bound": "alu", "frac": 2 / 3}, "work_per_launch": {"f16": [1 / 3] * 50},
            "accuracy_vs_fp64_oracle": {"a": err, "b": {"rel_err_max": 3e-7, "compared": 10}},
            "cluster_cut": [{"tau": 1e-3, "x": "y" * 500}], "footprint_kernels": {"disk": "z" * 500},
            "jacobian_clamp_and_sampling": {"x": "y" * 500},
            "glint_diffuse_16384": {"workload": "w" * 500, "projected_area": {"ms": 1 / 3, "triangles": 24863572700},
                                    "pndf": {"ms": 1 / 3}, "ggx_fit": {"x": [1 / 3] * 300},
                                    "served_stream": {"served_equals_plain_bitwise": True, "loads": [1] * 100}},
            "serving": {"four_maps": stream, "flake8192_only": stream, "wall_s": 1.0, "note": "n" * 100},
            "kernel_rooflines": {"families": {f"family{k}": {"ms": 1 / 3, "bound": "issue", "frac": 1 / 3, "kernels": ["k"] * 20}
                                              for k in range(8 + extra)}}}


@pytest.mark.parametrize("extra", [0, 200])
def test_line_is_short_and_keeps_the_measurement(bench, extra):
    line = full_line(bench, extra)
    text = json.dumps(bench.summary_line(line))
    assert len(text) <= bench.LINE_LIMIT and "\n" not in text
    got = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert got[k] == line[k], k
    if not extra:
        assert got["rel_err_max_vs_fp64_oracle"] == {"a": 2e-6, "b": 3e-7}
        assert got["serving"]["four_maps"]["loads"][0]["arm0"] == {"p50_ms": 0.333333, "p99_ms": 0.666667}
        assert got["glint_diffuse_16384"]["served_stream"] == {"served_equals_plain_bitwise": True}


def test_a_line_of_the_measurement_alone(bench):
    line = {k: v for k, v in full_line(bench).items() if k in ("metric", "value", "ms_per_step", "e2e", "config")}
    assert bench.summary_line(line) == line


def test_measured_traffic_decides_the_bound(bench, monkeypatch):
    monkeypatch.setattr(bench, "compute_peaks", lambda dev: {"issue": 1258.56, "fp32": 80.0, "fp64": 1.25, "sms": 152, "sm_mhz": 2070.0})
    monkeypatch.setattr(bench, "hbm_peak", lambda: (6000.0, "measured"))
    monkeypatch.setattr(bench, "committed_ncu_pct", lambda tag: None)
    monkeypatch.setattr(bench, "committed_profile_value", lambda key: 6e4)
    nq = bench.synth.FLAKE_8192["queries"]
    w = {"nodes": 10000 * nq, "leaf_blocks": 1200 * nq, "bytes": 1, "quads": 1, "tri_tests": 1, "hits": 1}
    monkeypatch.setattr(bench, "committed_traffic", lambda tag: 1.0e12)
    r = bench.traversal_roofline(None, w, nq=nq, kernel_ms=330.0, world=1)
    assert r["hbm"]["frac"] > r["issue"]["frac"] > r["hbm"]["measured_frac"]
    assert r["bound"] == "alu" and r["frac"] == r["issue"]["frac"]
    assert abs(r["hbm"]["measured_frac"] - 1.0e12 / 0.33 / 1e9 / 6000.0) < 1e-12
