"""The line that the default run of bench.py prints: the figures of every record, in a few kilobytes."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402

PROSE = "how it was measured, " * 40


def _full():
    roof = {"bound": "alu", "achieved": 2.6e11, "peak": 1.26e12, "unit": "warp-instructions/s", "frac": 0.2071,
            "traffic": None, "kernel": "k_scan_columns", "launch_ms": 0.0076, "note": PROSE, "timing": PROSE}
    runs = {arm: [{"seed": s, "time_s": 0.0067, "gens": 212, "gens_run": 216, "final": 5747, "evals": 161462}
                  for s in range(5)] for arm in ("plain", "learned")}
    learned = {"workload": PROSE, "target": 5747, "target_check": PROSE, "plain_time_s": 0.0067, "learned_time_s": 0.0023,
               "speedup_amortised": 2.9, "reached": {"plain": 3, "learned": 5}, "plain_ms_per_gen": 0.032,
               "learned_ms_per_gen": 0.1, "model": {"trained_on": PROSE}, "roofline": roof, "clocks": {}, "runs": runs}
    passes = [{"workload": "euclid10000", "p": p, "pop": 4096, "steps": 3000, "ms_per_pass": 0.138, "evals_per_s": 3e7,
               "roofline": dict(roof, traffic_frac=0.2), "roofline_issue": roof, "clocks": {}} for p in (10, 100, 1000)]
    return {"metric": bench.METRIC, "value": 1.1e8, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.157, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "int64",
            "data": "synthetic", "config": {"workload": "graph900", "description": "x" * 200, "n": 900, "m": 900, "p": 90},
            "evals": 349525, "best_cost": 1, "gpu_launches": 460, "roofline": roof,
            "roofline_alg_bytes": dict(roof, l2_bytes=1.0, pass_ms=0.02),
            "e2e": {"value": 9e7, "unit": bench.UNIT, "h2d_bytes_per_step": 162000.0, "d2h_bytes_per_step": 14.8,
                    "note": PROSE},
            "cpu_baseline": {"value": 72369.2, "unit": bench.UNIT, "how": "x" * 300},
            "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []}, "eval_euclid10000": passes,
            "learned": {n: learned for n in ("gmm5000_p500", "gmm5000_p50", "graph100")},
            "batched256": {"value": 1e8, "unit": "evals/s", "ms_per_step": 7.0, "steps": 20, "config": {"d": PROSE},
                           "roofline": roof, "eval_tile": {"groups": 4}}, "extra_s": 12.0}


def test_the_headline_keeps_every_contract_key_and_is_short():
    full = _full()
    line = bench.headline(full)
    assert len(json.dumps(full)) > 12000 and len(json.dumps(line)) < 4096
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "cpu_baseline", "evals"):
        assert line[key] == full[key], key
    assert set(line["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert line["roofline"]["frac"] == full["roofline"]["frac"] and line["roofline"]["bound"] == "alu"
    assert [r["ms_per_pass"] for r in line["eval_euclid10000"]] == [0.138] * 3
    assert line["learned"]["graph100"]["learned_time_s"] == 0.0023
    assert line["batched256"]["ms_per_step"] == 7.0


def test_a_run_without_the_extra_records():
    full = {k: v for k, v in _full().items() if k not in ("eval_euclid10000", "learned", "batched256", "extra_s")}
    full.update(n_gpus=8, cpu_baseline=None)
    line = bench.headline(full)
    assert line["n_gpus"] == 8 and "learned" not in line and line["cpu_baseline"] is None
