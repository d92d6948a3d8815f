"""The bench's line stays short enough for a reader that keeps only the last few kilobytes of its output: the
autotune tables go to stderr, and its numbers keep seven digits."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tables_are_split_off():
    sys.path.insert(0, ROOT)
    import bench
    row = {"tpa": 16, "list": "full", "block": 128, "vec": 1, "ms": 1.5547840595245361}
    line = {"value": 4049125258.123456, "steps": 20, "vs_baseline": None, "clocks": {"reasons": ["sw_power_cap"], "sm_mhz": 2062.5},
            "autotune": [row] * 36,
            "extras": {"lj": {"mixed": {"value": 1.0 / 3.0, "tpa": 1, "rebuilds": 8, "note": "long"}, "autotune": [row] * 72, "fp64_autotune": [row] * 72}}}
    short, rest = bench.split_tables(line)
    assert len(json.dumps(short)) < 400
    assert sorted(rest) == ["autotune", "extras", "extras/lj/autotune", "extras/lj/fp64_autotune"]
    assert rest["autotune"] == [row] * 36 and rest["extras"] is line["extras"]
    assert short["value"] == 4049125000.0 and short["steps"] == 20 and short["vs_baseline"] is None
    assert short["clocks"] == {"reasons": ["sw_power_cap"], "sm_mhz": 2062.5}
    assert short["extras"]["lj"]["mixed"] == {"value": 0.3333333, "tpa": 1}
