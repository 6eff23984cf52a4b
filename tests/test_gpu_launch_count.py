"""Kernel launches of one step: the reservoir branch counts its cells (1),
scans the counts (1 launch up to 2048 reservoir cells, 2 above) and writes its
particles (1)."""
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny,branch", [(12, 3), (1024, 3), (1025, 4)])
def test_launches_of_the_reservoir_branch(ny, branch):
    import paper_2506_23917_gb300 as sp

    n = []
    for inflow in (False, True):
        cfg, regions = W.box2d(nx=4, ny=ny, ppc=3.0, body=False, inflow=inflow)  # two reservoir layers of ny cells
        pos, vel = W.fill_regions(cfg, regions, 1)
        s = sp.Sim(cfg, sp.FP64, capacity=4 * vel.shape[1] + 1000)
        s.set_particles(0, pos, vel)
        s.step(1)
        s.sync()
        n.append(s.launches_per_step())
        s.close()
    assert n[1] - n[0] == branch
