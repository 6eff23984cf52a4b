"""FP32 state: the collision schedule changes no bit, also where a cell above
256 particles shares its batch with others (its sum is taken by the whole
warp, and one lane's FP32 pair stands for it) and above every staging size."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", ["tube", "cylinder"])
def test_fp32_schedule_changes_no_bit(shape):
    import paper_2506_23917_gb300 as sp

    if shape == "tube":  # 260 to 1100 per cell, hybrid cells
        cfg, regions = W.sod(ncell=96, ppc_left=520.0, lam_left=3e-3, n_steady=0)
        regions[1].update(n=0.5 * regions[0]["n"])
        steps = 60
    else:
        cfg, regions = W.cylinder(scale=0.2, ppc=60.0, n_steady=0)
        steps = 120
    pos, vel = W.fill_regions(cfg, regions, 7)
    ref = None
    for sched in ((864, 2), (1024, 4), (512, 4), (128, 8), (928, 2)):
        s = sp.Sim(cfg, sp.FP32, capacity=2 * vel.shape[1] + 100000)
        s.set_particles(0, pos, vel)
        s.set_schedule(*sched)
        s.step(steps)
        got = [*s.particles(0), s.moments(0, 1), s.sigc_max(0)]
        s.close()
        if ref is None:
            ref = got
        for x, y in zip(ref, got):
            assert np.array_equal(x, y), sched
