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


@pytest.mark.parametrize("launches,steps,spl,kernel", [
    (20, 20, 1, "step_kernel"), (24, 20, 1, "step_kernel"),   # FP16: counter bumps beside
    (10, 20, 2, "fused_step_kernel"), (12, 20, 2, "fused_step_kernel"),
    (160, 300, 2, "fused_step_kernel"),
    (5, 20, 4, "tile_step_kernel"), (9, 100, 11, "tile_step_kernel"), (27, 300, 11, "tile_step_kernel")])
def test_steps_per_launch_and_kernel(launches, steps, spl, kernel):
    """Small lattices advance 4 to 16 steps a launch: the mean, and their kernel."""
    assert bench.steps_per_launch(launches, steps) == spl
    assert bench.kernel_name("auto", "StoreF32", spl) == f"lbmp::{kernel}<StoreF32>"
