"""The benchmark's JSON line stays short enough to be read from the end of a run's output: no array with a value per frame
in it, and floats inside the blocks to six digits."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_compact():
    import bench

    rec = {k: [100_000_000 + 7 * i for i in range(100)] for k in "abcdefgh"}
    line = {"value": 170391562.22341052, "unit": "q", "stage_ms": {"fit": 23.524512345, "n": 100_000_693},
            "run": {"fit_ms_per_table": [22.76512345, 23.0]}, "vs_baseline": None, "ok": True, "reasons": ["a"] * 20,
            "other_configs": {"stream": {m: rec for m in ("exact", "scheduled")}}}
    out = bench.compact(line)
    assert len(json.dumps(line)) > 17_000 and len(json.dumps(out)) < 2_000
    s = out.pop("other_configs")["stream"]
    assert s["exact"]["a"] == {"mean_min_max_last": [1e8, 100_000_000, 100_000_693, 100_000_693]}
    assert sorted(s["scheduled"]) == sorted(rec)
    assert out == {"value": 170391562.22341052, "unit": "q", "stage_ms": {"fit": 23.5245, "n": 100_000_693},
                   "run": {"fit_ms_per_table": [22.7651, 23.0]}, "vs_baseline": None, "ok": True, "reasons": ["a"] * 20}
