"""A column pass over short columns keeps up with the other passes: at 4 x 1024 x 1024
its 16-column tiles of 16 threads are 131,000 blocks, so anything a block does besides its
columns shows.  All passes move the same bytes, in L2.  Measured on GB300: x-pass 23 us
and z-pass 11.5 us; with an early release of the next pass in each block 39 and 12 us."""
import pytest

pytestmark = pytest.mark.gpu


def test_short_column_pass_costs_no_more_than_its_tiles():
    import torch
    import paper_2202_12756_gb300 as fft3d
    plan = fft3d.Plan((4, 1024, 1024), torch.float32)
    buf = plan.empty_padded().uniform_(-1.0, 1.0)
    least = {}
    for _ in range(20):
        plan.set_profiling(True)
        for _ in range(3):
            plan.r2c_(buf)
            plan.c2r_(buf)
        torch.cuda.synchronize()
        for k in plan.profile_read():
            least[k["name"]] = min(least.get(k["name"], 1e9), k["total_ms"] / k["launches"])
        plan.set_profiling(False)
    # halfway (geometrically) between the two measured ratios, 2.0 and 3.3
    assert least["r2c.x"] <= 2.56 * least["r2c.z"], least
    assert least["c2r.x"] <= 2.56 * least["c2r.z"], least
