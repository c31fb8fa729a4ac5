"""The line that bench.py prints: short enough for a reader that keeps the last 3 KB of the output, whatever
the record holds, with every field that the benchmark's readers take; the whole record goes to standard
error."""
import json

import pytest


def record(filler):
    text = "words " * filler
    part = {"value": 1.23456789012e10, "unit": "points/s", "ms_per_step": 2.345678901, "steps": 20,
            "config": {"workload": "many_bubbles_l4-10", "leaves": 31265592, "l2": text, "launch": {"a": text}},
            "roofline": {"bound": "hbm", "kernel": text, "achieved": 2034.234567, "peak": 6781.8, "unit": "GB/s",
                         "frac": 0.29995, "traffic": None, "traffic_source": text},
            "cpu_baseline": {"value": 3188096.123, "unit": "points/s", "cores": 16, "kind": "oracle", "sample": text},
            "e2e": {"value": 6.12168e9, "unit": "points/s", "h2d_bytes_per_step": 1272000001,
                    "d2h_bytes_per_step": 1332249472, "ms_per_step": 8.4944, "pipeline": text},
            "parity": {"all_ok": True, "tolerance": 1e-5, "forms": {str(k): text for k in range(9)}},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"]}, "forms": {"x": text}}
    return dict(part, metric="points/s of " + "m" * 60, n_gpus=1, warmup=5, higher_is_better=True, scaling="weak",
                vs_baseline=None, dtype="f32", data="synthetic", gpu_launches=440,
                workloads={k: part for k in ("tiny", "single_bubble", "learned_index", "tracking")})


@pytest.mark.parametrize("filler", [0, 5, 40, 4000])
def test_line(filler, capsys):
    import bench
    out = record(filler)
    bench.report(out)
    got = capsys.readouterr()
    assert got.out.count("\n") == 1 and len(got.out) <= 2500
    line = json.loads(got.out)
    for k in ("metric", "unit", "n_gpus", "steps", "warmup", "higher_is_better", "scaling", "vs_baseline", "dtype", "data",
              "gpu_launches"):
        assert line[k] == out[k]
    for k in ("value", "ms_per_step"):
        assert line[k] == pytest.approx(out[k], rel=1e-6)
    for k in ("h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][k] == out["e2e"][k]
    assert line["e2e"]["value"] == pytest.approx(out["e2e"]["value"], rel=1e-6)
    assert line["clocks"] == out["clocks"] and line["config"]["workload"] == out["config"]["workload"]
    assert set(line["workloads"]) == set(out["workloads"])
    assert json.loads(got.err.split("[bench] record ", 1)[1]) == out


def test_a_failed_workload_keeps_its_error():
    import bench
    out = record(3)
    out["workloads"]["tiny"] = {"error": "ValueError: no", "wall_s": 1.0}
    assert bench.headline(out)["workloads"]["tiny"] == {"error": "ValueError: no"}
