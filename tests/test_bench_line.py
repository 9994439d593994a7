"""The benchmark's printed line: short enough for a reader that keeps the last 3000
characters of the output, with every key a reader of the metric needs; the record
that it is taken from keeps everything."""
import json

import bench


def block(n):
    return {"value": 1.2345678901234567e11, "unit": bench.UNIT, "ms_per_step": 8.320729827880859, "steps": 20,
            "e2e": {"value": 4.0636526021275276e10}, "detail": ["x" * 50] * n}


def test_line_is_short_and_complete():
    rec = dict(block(20), metric=bench.METRIC, n_gpus=1, warmup=5, higher_is_better=True, scaling="weak",
               vs_baseline=None, dtype="f32", data="synthetic", gpu_launches=760, newton_iterations_per_fit=1.11)
    rec["config"] = {"workload": "harris_512x256_v16", "grid": [512, 256], "precision": "f" * 140, "note": "n" * 150}
    rec["roofline"] = {"kernel": "v_pass", "bound": "hbm", "achieved": 2678.5714658263623, "peak": 6793.1, "unit": "GB/s",
                       "frac": 0.39430767482097456, "traffic": None, "peak_kind": "measured",
                       "algorithmic_bytes_per_launch": 4294967296}
    rec["phases_ms_per_step"] = {k: 1.2345678901234567 for k in ("fields", "fit_exchange", "fit_solve", "fluid", "v_pass", "xy_sweep")}
    rec["clocks"] = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 3}
    rec["e2e"] = {"value": 4.0636526021275276e10, "unit": bench.UNIT, "h2d_bytes_per_step": 4294967296,
                  "d2h_bytes_per_step": 4294967296, "steps": 20, "ms_per_step": 26.42307, "run_reported": "fastest of 8",
                  "runs_ms_per_step": [41.315582275390625] * 8}
    rec["mlp"] = {"newton_iterations_per_fit": 1.11, "fits_started_warm": 0.97, "cold_start": block(5)}
    rec["cpu_baseline"] = {"value": 1265584.0, "unit": bench.UNIT, "cores": 1, "kind": "oracle", "sample": "s" * 200}
    rec["fp64_form"] = dict(block(10), hbm_phases={"v_pass": 1})
    rec["newton_roofline"] = {"bound": "latency", "frac": 0.01, "unit": "GB/s", "evaluations": {}}
    rec["workloads"] = {n: block(60) for n in ("asym_1024x512_v12", "harris_128x64_v20", "landau_64x32")}
    line = bench.printed_line(rec)
    text = json.dumps(line)
    assert len(text) < 2900, len(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "roofline"):
        assert line[k] == rec[k]
    for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == rec["e2e"][k]
    assert set(line["workloads"]) == set(rec["workloads"])
    assert line["mlp"]["cold_start_ms_per_step"] == rec["mlp"]["cold_start"]["ms_per_step"]


def test_line_without_optional_blocks():
    line = bench.printed_line({"metric": bench.METRIC, "value": 1.0, "e2e": None, "mlp": None, "cpu_baseline": None})
    assert line == {"metric": bench.METRIC, "value": 1.0}
