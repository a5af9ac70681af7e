"""The batched benchmark's printed line: short enough for a log that keeps the last
3 kB of the output, with every key of the contract, whatever the number of
correlation classes and tuned (m, R)."""
import json

import bench


def record(steps=20, keys=55, classes=14):
    tune = {"%d,%d" % (41 + 20 * (i % 4), 10 + i // 4): {"path": 6, "option": (96, 128, 160)[i % 3], "candidates_ms": {
        "5/0": 0.3 + i / 7, "6/128": 0.4, "6/96": 1 / 3}} for i in range(keys)}
    roof = {"bound": "alu", "achieved": 19.29748844985635, "peak": 80.12369724391301, "unit": "TFLOP/s",
            "frac": 0.24084620547540167, "traffic": None, "kernel": "k_corr_fft (FP32 Fourier, Eq. 13) class 160",
            "launch_ms": 29.42902374267578, "peak_src": "p" * 120, "work": "w" * 120,
            "classes": [{"kernel": "k" * 30, "path": 6, "cls": 96 + i, "launches": 1, "ms": i + 1 / 3, "items": 23169,
                         "m": [41, 61], "R": [10, 40], "traffic": None, "achieved": 1 / 7, "frac": 1 / 3} for i in range(classes)]}
    form = {"value": 818594.2674720866, "ms_per_step": 146.1798655999999, "steps": steps, "sfoc_mpix_s": 17103.68241,
            "stage_ms_per_step": {k: 1 / 3 for k in "abcdefg"}, "roofline": roof, "matched_per_step": 119662,
            "gpu_launches": 820, "launches_per_step": 41.0, "first_call_s": 0.74, "graph": True, "autotune": tune}
    return {"metric": bench.METRIC, "value": form["value"], "unit": bench.UNIT, "n_gpus": 1, "steps": steps, "warmup": 5,
            "ms_per_step": form["ms_per_step"], "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic", "config": {"workload": "x" * 190, "l2": "y" * 90, "form": "bf16batch"},
            "roofline": roof, "cpu_baseline": {"value": 3.585269951279335, "sample": "z" * 160}, "gpu_launches": 820,
            "e2e": {"value": 8e5 / 3, "unit": "CP/s", "h2d_bytes_per_step": 2330240104, "d2h_bytes_per_step": 2961264,
                    "call": "c" * 90, "step_done_ms": [146.1] * steps, "sync_call_ms": [148.2] * steps},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "scope": "timed region"},
            "sfoc_mpix_s": 17103.68241, "stage_ms_per_step": form["stage_ms_per_step"], "parity": {"points": 4},
            "gathered": None, "forms": {f: dict(form) for f in ("bf16batch", "f32batch", "f32plain")},
            "bf16batch_over_f32plain": 18.399, "peaks": {"hbm_gbs": 6780.7, "src": "measured", "microbench": {"x": 1 / 3}},
            "errors": None}


def test_the_line_is_short_and_whole():
    full = record()
    assert len(json.dumps(full)) > 10000
    text = json.dumps(bench.short_line(full))
    assert len(text) < 3000
    line = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks"):
        assert k in line, k
    for k in ("bound", "achieved", "peak", "unit", "frac", "traffic"):
        assert k in line["roofline"], k
    assert abs(line["value"] / full["value"] - 1) < 1e-5 and line["value"] == line["forms"]["bf16batch"]["value"]
    assert line["e2e"]["h2d_bytes_per_step"] == 2330240104
    assert [c["cls"] for c in line["roofline"]["classes"]] == [109, 108]
    assert sum(line["forms"]["f32batch"]["autotune"].values()) == 55


def test_the_longest_runs_still_fit():
    assert len(json.dumps(bench.short_line(record(steps=500, keys=200, classes=40)))) < 3000


def test_fast_reports_what_the_kernel_executes_beside_the_definition():
    """2048 x 2048 in 24.6 us: the score at every pixel, most of which the quick test
    spares, and the quick test itself."""
    r = bench.fast_roofline(0.0246, 2048, 2048, 6780.0)
    assert "spared" in r["work"] and r["executed_floor_ops"] == 24
    assert abs(r["executed_floor_frac"] * r["peak"] * 1e12 / (24 * 2048 * 2048 / 24.6e-6) - 1) < 1e-9
    assert r["executed_floor_frac"] < r["frac"]
