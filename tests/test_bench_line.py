"""The headline that bench.py prints is one short line: every key a reader of the
headline needs, and none of the long records."""
import json

import bench


def _record():
    return {"metric": bench.METRIC, "value": 95214.4, "unit": "MLUPS", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.17621, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 4025.0, "unit": "MLUPS", "h2d_bytes_per_step": 603979776,
                    "d2h_bytes_per_step": 603979816}, "gpu_launches": 20,
            "config": {"workload": "tgv_bgk_4096x4096", "nx": 4096, "ny": 4096},
            "timing": {"runs": 5, "run_ms_per_step": [0.176] * 400, "headline": "median run"},
            "tau_sweep": [{"tau": 0.8, "mlups": 1.0}] * 100,
            "cpu_baseline": {"value": 5.8, "unit": "MLUPS", "gnn": {"value": 1.0, "note": "x" * 3000}},
            "gnn": {"xavier": {"workload": "tgv_gnn_1024x1024", "mlups_gnn": 1932.4, "ms_per_step_gnn": 0.5426,
                               "l2_error_gnn": float("nan")},
                    "tgv_tables": {"rows": list(range(20000))}}}


def test_headline_is_short_and_whole():
    rec = _record()
    h = bench.headline(rec)
    line = json.dumps(bench._finite(h), allow_nan=False)
    assert "\n" not in line and len(line) < 2500 < len(json.dumps(bench._finite(rec)))
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "e2e", "clocks", "gpu_launches"):
        assert h[k] == rec[k]
    assert h["gnn"]["xavier"] == {"workload": "tgv_gnn_1024x1024", "mlups_gnn": 1932.4, "ms_per_step_gnn": 0.5426}
    assert rec["gnn"]["tgv_tables"]["rows"]  # the record itself is left whole


def test_reference_line_passes_unchanged():
    ref = {"impl": "reference", "value": 5.8, "cpu_baseline": {"value": 5.8, "unit": "MLUPS"}}
    assert bench.headline(ref) == ref
