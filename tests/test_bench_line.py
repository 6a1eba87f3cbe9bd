"""The line that bench.py prints stays short enough to be read from the end of a run's output, whatever the record
holds, and keeps the headline's keys."""
from __future__ import annotations

import json

import pytest
from test_bench_host import load_bench


def record(configs):
    long = {"what": "x" * 400, "value": 1.23456789012345e13}
    call = {"ms_per_step": 0.0651234567, "frames_per_s": 4.6123456789e9, "outputs_equal": True, "what": "y" * 300,
            "roofline": {"bound": "hbm", "achieved": 1289.123456, "frac": 0.19012345, "note": "z" * 300},
            "e2e": {"value": 6.4e8, "unit": "frames/s", "ms_per_step": 0.46}}
    rec = {"metric": "TEP syndrome checks/s & frames/s per GB300; p50/p99 decode latency", "value": 4.4123456789e13,
           "unit": "checks/s", "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 2.1723456789,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u32",
           "data": "synthetic (seeded random polar codewords over AWGN)",
           "config": {"workload": "polar N=128 K=64, 16-QAM Gray, Eb/N0 6/8/10 dB x 100000 frames, S=10, cap 2^20",
                      "tiles": [0, 0, 1, 4], "l2": "flushed before every timed step (256 MiB write)"},
           "frames_per_s": 1.38e8, "bler": 0.1, "latency_ms": {"p50": 2.17, "p99": 2.2, "what": "w" * 50},
           "e2e": {"value": 4.1e13, "unit": "checks/s", "h2d_bytes_per_step": 76800000, "d2h_bytes_per_step": 6300000,
                   "ms_per_step": 2.36, "api": "a" * 100}, "roofline": {**long, "bound": "smem", "frac": 0.8},
           "default_call": call, "demod": {"ms": 0.033, "frac": 0.83, "timing": "t" * 200}, "solve": long,
           "cpu_baseline": {"value": 5.1e7, "unit": "checks/s", "cores": 16, "kind": "oracle", "sample": "s" * 90},
           "gpu_launches": 40, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 9}}
    if configs:
        rec["configs"] = {f"c{i}": {**record(0), "latency_us": {"p50": 112.7, "p99": 169.4, "max": 268.0}}
                          for i in range(configs)}
    return rec


@pytest.mark.parametrize("configs", [0, 1, 5, 40])
def test_line_is_short_and_whole(configs):
    bench = load_bench()
    rec = record(configs)
    text = json.dumps(bench.short_line(rec))
    assert len(text) <= 2600
    out = json.loads(text)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert k in out, k
    assert out["value"] == pytest.approx(rec["value"], rel=1e-5) and out["unit"] == "checks/s"
    assert set(out["e2e"]) >= {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert out["default_call"]["frames_per_s"] == pytest.approx(4.6123456789e9, rel=1e-5)
    assert len(out["configs"]) == min(configs, 5) or configs == 40


def test_bit_level_record():
    """The bit-level workload has no default call, demodulation or search roofline beside it."""
    bench = load_bench()
    rec = record(0)
    for k in ("default_call", "demod", "roofline"):
        rec[k] = None
    out = bench.short_line(rec)
    assert out["value"] == pytest.approx(rec["value"], rel=1e-5) and out["default_call"] is None
