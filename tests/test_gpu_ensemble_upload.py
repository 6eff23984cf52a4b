"""Uploads into a context of several instances: the instance of each particle
needs no memory of its own per slot, and a restart after any number of steps
gives each instance the bits of a context of its own."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_slots_cost_the_same_with_several_instances():
    import torch

    import paper_2506_23917_gb300 as sp

    cap = 1 << 24
    used = []
    for n_inst in (1, 2):
        cfgs = [W.sod(ncell=100, ppc_left=10.0)[0] for _ in range(n_inst)]
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        s = sp.Sim(cfgs, sp.FP32, capacity=cap)
        used.append(before - torch.cuda.mem_get_info()[0])
        s.close()
    assert used[0] >= 40 * cap  # (positions and velocities twice, keys twice, the permutation)
    assert abs(used[1] - used[0]) < cap  # below one byte per slot


@pytest.mark.parametrize("prec", ["FP32", "FP64"])
@pytest.mark.parametrize("kind", ["tube", "box2d", "ogrid"])
def test_restart_of_an_ensemble(kind, prec):
    import paper_2506_23917_gb300 as sp

    flows = []
    for i in range(3):
        if kind == "tube":
            cfg, regions = W.sod(ncell=20 + 13 * i, ppc_left=30.0 + 7 * i, n_steady=0)
        elif kind == "box2d":
            cfg, regions = W.box2d(nx=12 + 3 * i, ppc=12.0)
        else:
            cfg, regions = W.ogrid_box(nr=6 + i, nt=12 + i, ppc=10.0)
        cfg = dict(cfg, seed=5 + i)
        flows.append((cfg, *W.fill_regions(cfg, regions, 20 + i), *W.fill_regions(cfg, regions, 40 + i)))
    total = sum(f[2].shape[1] for f in flows)
    s = sp.Sim([f[0] for f in flows], getattr(sp, prec), capacity=4 * total + 30000)
    alone = [sp.Sim(f[0], getattr(sp, prec), capacity=4 * f[2].shape[1] + 10000) for f in flows]
    for again in (0, 1):
        for i, f in enumerate(flows):
            s.set_particles(i, f[1 + 2 * again], f[2 + 2 * again])
            alone[i].set_particles(0, f[1 + 2 * again], f[2 + 2 * again])
        for x in (s, *alone):
            x.step(3)  # (odd: the restart goes into the other buffers)
    for i, x in enumerate(alone):
        for p, q in zip(s.particles(i), x.particles(0)):
            assert np.array_equal(p, q), (kind, prec, i)
        assert np.array_equal(s.moments(i, 0), x.moments(0, 0), equal_nan=True)
        x.close()
    s.close()
