"""bench.py's reading of how many steps a launch advanced (no GPU needed)."""
import json
import os

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("storage", ["fp16", "fp32"])
def test_batch_traffic_is_of_launches_of_as_many_steps(storage):
    """Figures captured on launches of two steps say nothing about a run of
    single steps on the same instances."""
    with open(os.path.join(ROOT, "profiles", "step_traffic.json")) as fh:
        e = json.load(fh)[f"batch_{storage}"]
    assert e["steps_per_launch"] == 2
    r = dict(ms=0.71 * 300, nodes=e["nodes"], bpu=44.0, staged=True)
    pairs = bench.batch_roofline(dict(r, launches=160), 300, 6795.8, "measured", storage)
    assert pairs["traffic"] == e["dram_bytes_per_launch"] and pairs["steps_per_launch"] == 2
    single = bench.batch_roofline(dict(r, launches=310), 300, 6795.8, "measured", storage)
    assert single["traffic"] is None and single["achieved_dram"] is None
