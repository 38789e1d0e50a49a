"""The instruction-issue roofline that bench.py reports for the double pair."""
import math

import bench


def test_issue_roofline_arithmetic():
    stats = [{"name": "r2c.y", "total_ms": 16.0, "launches": 2}, {"name": "c2r.z", "total_ms": 10.0, "launches": 2}]
    units = 1024 * 1024 * 513
    r = bench.issue_roofline(stats, {"r2c.y": 12.5}, 152, 2070.0, units)
    assert r["kernel"] == "r2c.y" and r["avg_launch_ms"] == 8.0
    assert r["peak"] == round(152 * 4 * 2.07, 1)  # G warp instructions/s
    assert math.isclose(r["achieved"], 12.5 * units / 8e-3 / 1e9, rel_tol=1e-3)
    assert math.isclose(r["frac"], r["achieved"] / (152 * 4 * 2.07), rel_tol=1e-3)
    # not counted on these sources, or no clock samples: no fraction
    assert bench.issue_roofline(stats, None, 152, 2070.0, units)["frac"] is None
    assert bench.issue_roofline(stats, {"r2c.y": 12.5}, 152, None, units)["frac"] is None
    assert bench.issue_roofline([], None, 152, 2070.0, units) is None
