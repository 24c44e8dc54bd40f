"""The benchmark's result line (CPU only): complete where it is read by others, and short."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_line_keeps_the_headline_and_the_figures_of_the_rows():
    headline = {"metric": "m", "value": 475.123456789, "unit": "apps/s", "n_gpus": 1, "steps": 20, "warmup": 5,
                "ms_per_step": 2.1, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
                "dtype": "bf16x3 (f32 accumulate)", "data": "synthetic", "config": {"grid": [256, 256, 256]},
                "roofline": {"frac": 0.4, "stage_ms_per_app": [1.4, 0.5]}, "gpu_launches": 4,
                "e2e": {"value": 450.0, "unit": "apps/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
                "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "cpu_baseline": {"value": 0.08}}
    entry = {"kind": "bf16x3_tile_width", "key": [0, 128, 0], "value": 128, "ms": 1.1, "ms_default": 1.1}
    rows = {"autotune": {"full": [entry] * 40, "cp": [entry] * 4},
            "cp": {"value": 85949.14416653693, "unit": "apps/s", "rel_l2": 5.6e-7, "roofline": {"frac": 0.23}},
            "forms_full": {"fp32": {"apps_per_s": 66.2, "rel_l2": 1.1e-6}},
            "uneven_batch": {"value": 2678.3, "rel_l2_sampled_max": 4.2e-6, "note": "x" * 400},
            "energy_study_uniform_cube": {"sizes": [64, 128], "rows": [{"n": 64, "energy": 0.166}] * 60}}
    record = dict(headline, **rows)
    line = bench.line_of(record)
    assert {k: line[k] for k in headline} == headline
    assert line["cp"] == {"value": 85949.1, "rel_l2": 5.6e-7, "roofline": {"frac": 0.23}}
    assert line["forms_full"] == {"fp32": {"apps_per_s": 66.2, "rel_l2": 1.1e-6}}
    assert line["uneven_batch"] == {"value": 2678.3, "rel_l2_sampled_max": 4.2e-6}
    assert "autotune" not in line and "energy_study_uniform_cube" not in line
    assert len(json.dumps(record)) > 6000 > 3 * len(json.dumps(line))
