"""Ensembles whose instances differ in cost per particle by orders of
magnitude: batches end early where their cells are dear, which changes no bit."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _ensemble(kns, n):
    return [W.homogeneous_box(m, kn, seed=i + 1, n_steady=0) for i, (kn, m) in enumerate(zip(kns, n))]


def _run(ins, prec, steps, sched=None):
    import paper_2506_23917_gb300 as sp

    s = sp.Sim([c for c, _, _ in ins], getattr(sp, prec), capacity=sum(v.shape[1] for _, _, v in ins) + 64)
    for i, (_, p, v) in enumerate(ins):
        s.set_particles(i, p, v)
    if sched:
        s.set_schedule(*sched)
    s.step(steps)
    s.sync()
    out = [x for i in range(len(ins)) for x in (*s.particles(i), s.moments(i, 1))]
    s.close()
    return out


@pytest.mark.parametrize("prec", ["FP32", "FP64", "FP32_CELL32"])
def test_the_partition_changes_no_bit(prec):
    ins = _ensemble([3e-4, 1.0, 2e-3, 0.3, 1e-2], [3000, 2500, 1700, 40, 900])
    together = _run(ins, prec, 12)
    apart = [x for one in ins for x in _run([one], prec, 12)]
    other = _run(ins, prec, 12, sched=(128, 4))
    for x, y, z in zip(together, apart, other):
        assert np.array_equal(x, y) and np.array_equal(x, z)
