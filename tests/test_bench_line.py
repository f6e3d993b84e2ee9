"""The line bench.py prints last stays short and strict JSON whatever the legs hold; the
whole record goes to stderr."""
import json

import bench


def _record():
    long = [{"job": k, "rel_l2_rho": 1e-5 / (k + 1), "storage": "f32"} for k in range(200)]
    return {
        "metric": "m", "value": 1.5e5, "unit": "MLUPS", "n_gpus": 1, "steps": 3, "warmup": 3,
        "ms_per_step": 100.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f32", "data": "synthetic", "config": bench.config_dict(bench.workload_set(5000)),
        "parallelism": "single",
        "roofline": {"bound": "l2", "achieved": 1.0, "peak": 2.0, "frac": 0.5, "unit": "GB/s",
                     "kernel": bench.STEP_KERNEL["march"], "peak_source": "x" * 500},
        "roofline_large": {"bound": "hbm", "frac": 0.8, "one_cell_per_thread": {"mlups": 1.0}},
        "cpu_baseline": {"value": 140.0, "unit": "MLUPS", "cores": 16, "kind": "oracle",
                         "sample": "s", "timings": long},
        "e2e": {"value": 1.4e5, "unit": "MLUPS", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, "gpu_launches": 5000,
        "reflected_energy": {"I": float("nan"), "II": 2e-4},
        "divergent_solves": {"I": "grows " * 50}, "roofline_sweep": long,
        "serving": {"served": {"solves_per_s": 22.0, "p99_s": float("inf")}, "oracle_sample": long},
        "parity": {"cases": long, "missed": long[:3]}, "batched": {"mlups": 1.4e5}, "d3q15": None,
    }


def test_the_line_is_short_strict_json_with_every_headline_key():
    record = _record()
    assert len(json.dumps(record)) > 20000
    text = json.dumps(bench.summary_line(record), allow_nan=False)
    assert len(text) < 3000 and "\n" not in text
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
                "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
                "clocks", "gpu_launches", "parallelism"):
        assert line[key] == record[key]
    assert line["roofline"]["frac"] == 0.5 and line["reflected_energy"] == {"I": None, "II": 2e-4}
    assert line["legs"]["parity_cases"] == 200 and line["legs"]["parity_missed"] == 3
    assert line["legs"]["served_solves_per_s"] == 22.0 and line["legs"]["served_p99_s"] is None


def test_a_run_without_legs():
    record = {k: v for k, v in _record().items() if k in ("metric", "value", "config")}
    assert bench.summary_line(record | {"parity": None, "serving": None})["value"] == 1.5e5
    assert json.loads(json.dumps(bench.finite(_record()), allow_nan=False))
