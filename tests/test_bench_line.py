"""The bench's printed line, on the CPU: the contract's keys, and short enough to
survive a reader that keeps the last 3,000 characters of a program's output, with
every optional record present."""
import json

import bench


def full_record():
    x = 1382.9123456789012
    e2e = {"value": x, "unit": "GCUPS", "h2d_bytes_per_step": 110_012_345, "d2h_bytes_per_step": 123_456_789}
    rec = {
        "metric": bench.METRIC, "value": x, "unit": "GCUPS", "n_gpus": 8, "steps": 20, "warmup": 5,
        "ms_per_step": x, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "i32|i16x2 (exact integer)", "data": "synthetic",
        "config": {"workload": "long-reads-10k-zdrop", "pairs": 100_000, "cells_per_step": 30_250_000_000,
                   "mode": bench.WORKLOAD_DESC["long-reads-10k"], "precision": "auto", "pairs_i16x2": 100_000,
                   "pairs_sweep_i16x2": 100_000, "pairs_sweep_rerun_i32": 100_000,
                   "l2": "flushed between timed steps (512 MB write)", "parallelism": "replica x8"},
        "plain_per_pair": {"pairs": 4000, "gcups_plain": x, "gcups_batched_same_pairs": x, "ms_plain": x},
        "plain_long_per_pair": {"pairs": 400, "gcups": x, "call": "c" * 200},
        "step_ms": [x] * 2000, "phases_ms": {k: x for k in ("forward", "walk", "step", "validate", "place")},
        "autotune_ns_per_warp_step": {f"i16x2 R={r}": x for r in range(40)},
        "roofline": {"bound": "alu", "kernel": "k_xdrop (antidiagonal sweep)", "achieved": x, "peak": x,
                     "unit": "Tops/s", "frac": x, "traffic": x, "traffic_unit": "t" * 300, "probe": [x] * 5},
        "e2e": e2e, "gpu_launches": 12, "wall_s_timed": x,
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 12345, "power_w_max": 1379.76,
                   "reasons": ["hw_slowdown", "hw_thermal_slowdown", "sw_power_cap", "sw_thermal_slowdown"]},
        "graph": {"value": x, "unit": "GCUPS", "ms_per_step": x, "call": "c" * 200, "status": 0},
        "search": {"rows": [{"x": x}] * 100}, "fold": {"rows": [{"x": x}] * 100},
        "serving": {"capacity_gcups": x, "load_frac_of_capacity": 0.7, "p50_ms": x, "p99_ms": x, "refused": 123,
                    "per_kind": {"sw_protein": [x] * 50},
                    "fixed_rate": {"offered_rate_hz": 900.0, "requests": 12345, "p50_ms": x, "p99_ms": x}},
        "cpu_baseline": {"value": x, "unit": "GCUPS", "cores": 128, "kind": "oracle", "sample": "s" * 300},
    }
    rec["configs"] = {w: dict(rec) for w in ("short-dna-1k", "long-reads-10k", "long-pair-1m")}
    return rec


def test_printed_line_is_short_and_whole():
    rec = full_record()
    line = bench.printed_line(rec)
    assert "\n" not in line and len(line) <= 2900, len(line)
    d = json.loads(line)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks"):
        assert key in d, key
    assert abs(d["value"] / rec["value"] - 1) < 1e-5
    assert d["e2e"]["h2d_bytes_per_step"] == 110_012_345 and d["config"] == rec["config"]
    assert set(d["configs"]) == set(rec["configs"])


def test_printed_line_without_the_optional_records():
    rec = full_record()
    for key in ("plain_per_pair", "plain_long_per_pair", "graph", "serving", "configs", "cpu_baseline"):
        rec.pop(key, None)
    rec["plain_per_pair"] = None
    d = json.loads(bench.printed_line(rec))
    assert "serving" not in d and d["clocks"]["sm_mhz"] == 2070.0
