"""The line that bench.py prints: the contract's keys, in at most 1500 characters, from a full set of measurements
with numbers of full length and every optional part present (CPU only)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_headline_is_short_and_complete():
    sys.path.insert(0, ROOT)
    import bench
    x = 2916478149.6064863
    err = dict.fromkeys(("rho", "rho_u", "rho_v", "rho_w", "E"), 1.3861714879856228e-08)
    sweep = {f"p{p}": {"n_edge": 64, "n_points": 16777216, "fp64": x, "mixed": x, "mixed_vf32": x, "mixed_kernels": {}}
             for p in range(3, 8)}
    full = {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 8, "steps": 100, "warmup": 10,
            "ms_per_step": 45.123456789012345, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32x2+f64", "data": "synthetic", "config": bench.config("mixed"),
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 12345},
            "e2e": {"value": x, "unit": bench.UNIT, "runs": [x] * 3, "h2d_bytes_per_step": 1310720000,
                    "d2h_bytes_per_step": 1310720000},
            "gpu_launches": 1600, "kernels": {"volume": {"avg_ms": x}},
            "roofline": {"bound": "alu", "kernel": "interp_faces", "achieved": 4.123456789, "peak": 6.52345678, "unit": "TFLOP/s",
                         "frac": 0.63456789, "traffic": None, "peak_source": "x" * 300},
            "error_vs_fp64": {"max_rel": err, "l2_rel": err}, "fp64": {"value": x}, "fp32_viscous_branch": {"value": x},
            "p_sweep_updates_per_s": sweep, "ensemble_64_vortex": {"fp64": {"updates_per_s": x}},
            "cpu_baseline": {"value": 1466712.4051916183, "unit": "updates/s", "cores": 144, "kind": "oracle",
                             "sample": "y" * 200, "single_thread": {}}}
    text = json.dumps(bench.headline(full))
    assert len(text) <= 1500, len(text)
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert k in line
    assert abs(line["value"] - x) <= 1e-6 * x and line["config"] == full["config"] and line["clocks"] == full["clocks"]
    assert set(line["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert sorted(line["updates_per_s"]) == ["p3", "p4", "p5", "p6", "p7"]
    # Without the optional measurements.
    bare = {k: v for k, v in full.items() if k != "cpu_baseline"}
    bare["p_sweep_updates_per_s"] = {}
    assert "cpu_baseline" not in bench.headline(bare)
