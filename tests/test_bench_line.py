"""The bench's line stays short: a reader may keep only the last few KB of the output."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_auxiliary_records_shrink_to_their_headlines():
    record = {"ms_per_step": 1.25, "value": 2.0e9, "setup_ms": {"stages": {f"stage{i}": 1.0 for i in range(200)}}}
    assert bench.brief(record) == {"ms_per_step": 1.25, "value": 2.0e9}
    assert len(json.dumps({k: bench.brief(record) for k in ("c1", "c2", "c3", "c4", "offsurface_c5")})) < 500
    assert bench.brief({"error": "no device"}) == {"error": "no device"}
