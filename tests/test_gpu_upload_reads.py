"""Uploads straight into the state buffers (one instance, the context's own
type) against staged ones, and field reads into mapped page-locked memory
against reads through the device buffer: the same bits."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _flow(kind):
    cfg, regions = {"1d": lambda: W.sod(ncell=70, ppc_left=37.0, n_steady=0),
                    "2d": lambda: W.box2d(),
                    "ogrid": lambda: W.ogrid_box(),
                    "3d": lambda: W.box3d()}[kind]()
    return cfg, *W.fill_regions(cfg, regions, 4)


@pytest.mark.parametrize("prec", ["FP32", "FP64", "FP32_CELL32"])
@pytest.mark.parametrize("kind", ["1d", "2d", "ogrid", "3d"])
def test_direct_and_staged_uploads_agree(kind, prec):
    import torch

    import paper_2506_23917_gb300 as sp

    cfg, pos, vel = _flow(kind)
    pos, vel = pos.astype(np.float32).astype(np.float64), vel.astype(np.float32).astype(np.float64)
    got = []
    for f32 in (False, True):  # one of the two is the context's own type
        s = sp.Sim(cfg, getattr(sp, prec), capacity=3 * vel.shape[1] + 4096)
        for n in (vel.shape[1], vel.shape[1] - 33):  # a second upload replaces the first, steps in between
            put = s.set_particles_f32 if f32 else s.set_particles
            put(0, pos[:, :n], vel[:, :n])
            s.step(3)
        out = [*s.particles(0), np.array([s.dt(0)]), s.sigc_max(0)]
        for kind_ in (0, 1):
            paged = s.moments(0, kind_)
            pinned = torch.zeros(paged.shape, dtype=torch.float64).pin_memory()
            s.moments_into(0, kind_, pinned.data_ptr())
            assert np.array_equal(paged, pinned.numpy())
            out.append(paged)
        s.close()
        got.append(out)
    for x, y in zip(*got):
        assert np.array_equal(x, y)


def test_a_state_without_pairs_is_refused():
    import paper_2506_23917_gb300 as sp

    cfg, _ = W.sod(ncell=8, ppc_left=10.0)
    s = sp.Sim(cfg, sp.FP64, capacity=64)
    s.set_particles(0, np.array([[0.1]]), np.ones((3, 1)))  # one particle: no time step
    with pytest.raises(sp.SpError):
        s.step(1)
    s.set_particles(0, np.array([[0.1, 0.11]]), np.array([[1.0, 2.0], [0.0, 1.0], [0.0, 0.0]]))
    s.step(2)
    assert s.count(0) == 2
    s.close()
