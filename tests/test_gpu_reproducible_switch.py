"""sp_set_reproducible off and on again: switching it on puts the current
state in source order, so that a run switched off and on at once is, bit for
bit, one that never was."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["FP32", "FP32_CELL32"])
@pytest.mark.parametrize("kind", ["box", "cylinder", "subcells", "jet"])
def test_off_and_on_at_once(kind, prec):
    import paper_2506_23917_gb300 as sp

    if kind == "box":
        cfg, pos, vel = W.homogeneous_box(6000, 1e-2, ppc=700.0, n_steady=0)
    else:
        cfg, regions = (W.jet(scale=0.1, ppc=200.0, plenum=1.0, n_steady=0) if kind == "jet"
                        else W.cylinder(scale=0.1, ppc=30.0, n_steady=0))
        if kind == "subcells":
            cfg["subcells"] = 2
        pos, vel = W.fill_regions(cfg, regions, 5)
    sims = [sp.Sim(cfg, getattr(sp, prec), capacity=3 * vel.shape[1] + 200000) for _ in range(2)]
    for s in sims:
        s.set_particles(0, pos, vel)
        s.step(7)
    a, b = sims
    b.set_reproducible(False)
    b.set_reproducible(True)
    for _ in range(2):
        assert np.array_equal(a.moments(0, 0), b.moments(0, 0), equal_nan=True)
        for s in sims:
            s.step(3)
    for x, y in zip((*a.particles(0), a.moments(0, 1)), (*b.particles(0), b.moments(0, 1))):
        assert np.array_equal(x, y)
    # after steps in scatter order: the state that is ordered is the current
    # one, so that from here on the run repeats
    b.set_reproducible(False)
    b.step(4)
    b.set_reproducible(True)
    p, v, _ = b.particles(0)
    f = b.moments(0, 0)
    assert np.array_equal(f, b.moments(0, 0), equal_nan=True)
    c = sp.Sim(cfg, getattr(sp, prec), capacity=3 * vel.shape[1] + 200000)
    c.set_particles(0, p, v)  # (the particles in source order: the same order within each cell)
    assert np.array_equal(f, c.moments(0, 0), equal_nan=True)
    for s in (*sims, c):
        s.close()
