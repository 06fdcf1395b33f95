"""The line bench.py prints for its default run: short enough to survive a log of which 3 KB are
kept, with the contract's keys and the values of the full record."""

import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def _full():
    x = 1234.567890123456
    form = {"mlups": x, "mlups_per_gpu": x, "ms_per_step": x, "storage": "f16", "hbm_gbs_algorithmic": x,
            "hbm_frac_of_measured": x, "fp32_roofline_frac": x, "unstable": False,
            "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []}}
    text = "a note of some length " * 12
    hbm = {"achieved": x, "peak": x, "unit": "GB/s", "frac": x, "peak_source": text, "algorithmic_bytes_per_cell": 108}
    roof = {"bound": "tensor", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "traffic": x,
            "traffic_source": text, "kernel": "fused pull-stream-collide step (one launch per step)", "peak_source": text,
            "algorithmic_flops_per_cell": 47920, "useful_flops_per_cell": 90240, "achieved_useful": x, "frac_useful": x,
            "mma_flops_per_cell": 184320, "achieved_mma": x, "frac_mma": x, "hbm": hbm}
    return {"metric": bench.METRIC, "value": x, "unit": "MLUPS", "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": x,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32 collision, f16 storage, bf16 net", "data": "synthetic",
            "config": {"workload": "TGV 256^3 Re1600 NCO (27-20-20-4, seed-0 Kaiming weights), form=mixed", "n": 256,
                       "re": 1600.0, "nu": x, "u0": 0.05, "parallelism": "replicas x1",
                       "l2": "state larger than L2 (no flush needed)"},
            "roofline": roof,
            "cpu_baseline": {"value": x, "unit": "MLUPS", "cores": 16, "kind": "oracle", "sample": text[:120], "seconds": x,
                             "mlups_by_grid_and_threads": {str(k): text for k in range(9)}},
            "e2e": {"value": x, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 8, "note": text,
                    "repetitions_s": [x] * 3},
            "gpu_launches": 20, "clocks": form["clocks"], "forms": {f: dict(form) for f in bench.FORMS},
            "precision": {str(k): x for k in range(400)}}


def test_headline_is_short_and_complete():
    full = _full()
    text = json.dumps(bench.headline(full))
    assert len(text) <= 2900
    got = json.loads(text)
    assert got["value"] == full["value"] and got["ms_per_step"] == full["ms_per_step"]
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
              "gpu_launches", "clocks"):
        assert got[k] == full[k], k
    for k in ("bound", "achieved", "peak", "unit", "frac", "traffic"):
        assert k in got["roofline"], k
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert k in got["e2e"], k
    assert set(got["forms"]) == set(bench.FORMS)


def test_headline_keeps_what_was_not_run():
    full = dict(_full(), e2e=None, cpu_baseline=None, forms={"mixed": {"unavailable": "out of memory"}})
    got = bench.headline(full)
    assert got["e2e"] is None and got["cpu_baseline"] is None
    assert got["forms"] == {"mixed": {"unavailable": "out of memory"}}
