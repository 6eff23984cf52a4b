"""Moments of an FP64 state: 4 lanes per cell up to 128 particles, a warp
above.  Cells at the edges of the lane counts against 64-bit (longdouble)
sums; a cell's fields do not depend on the cells around it; the read of a
dense cell does not run on four lanes."""
import numpy as np
import pytest

from paper_2506_23917_gb300 import workloads as W

pytestmark = pytest.mark.gpu
SIZES = [5, 0, 1, 2, 3, 4, 31, 32, 33, 127, 128, 129, 130, 255, 256, 257, 4, 1023, 1024, 1025, 5000, 2, 128, 129]


def _flow(sizes, seed=2):
    """A 1-D row of unit cells holding the given particle counts, in random order."""
    cfg, _, _ = W.huge_cells((100,))
    cfg = dict(cfg, n=[len(sizes), 1, 1], hi=[float(len(sizes)), 1.0, 1.0], dt_fixed=1e-3)
    rng = np.random.Generator(np.random.PCG64(seed))
    cell = np.repeat(np.arange(len(sizes)), sizes)
    pos = (cell + rng.uniform(0.01, 0.99, len(cell)))[None]
    vel = rng.normal(0, 1, (3, len(cell))) + np.array([3.0, -1.0, 0.0])[:, None] + rng.exponential(1.0, (3, len(cell)))
    order = rng.permutation(len(cell))
    return cfg, np.ascontiguousarray(pos[:, order]), np.ascontiguousarray(vel[:, order]), cell[order]


def _fields(cfg, pos, vel, prec="FP64"):
    import paper_2506_23917_gb300 as sp

    s = sp.Sim(cfg, getattr(sp, prec), capacity=vel.shape[1] + 16)
    s.set_particles(0, pos, vel)
    f = s.moments(0, 0)
    s.close()
    return f


def test_moments_at_the_lane_counts():
    """A lane adds up to ceil(N / 4) + 6 terms one after another, each
    addition with a relative error of 2^-53 of the partial sum (at most the
    sum of the magnitudes), and each term takes up to 8 roundings more."""
    cfg, pos, vel, cell = _flow(SIZES)
    f = _fields(cfg, pos, vel)
    for k, n in enumerate(SIZES):
        assert f[0, k] == n
        if n == 0:
            continue
        c = vel[:, cell == k].astype(np.longdouble)
        u = c.mean(1)
        eps = (np.ceil(n / 4) + 14) * 2.0**-53
        assert np.all(np.abs(f[2:5, k] - u) <= eps * np.abs(c).mean(1)), (k, n)
        if n < 2:
            continue
        C = c - u[:, None]
        c2 = (C * C).sum(0)
        du = eps * np.abs(c).mean(1).max()  # (the shift's error enters squared, and the terms' to first order)
        T = c2.sum() / (3 * cfg["R"] * (n - 1))
        assert abs(f[5, k] - T) <= (eps + 4 * du / np.sqrt(c2.mean())) * T, (k, n)
        if n < 3:
            continue
        fq = 0.5 * n / ((n - 1) * (n - 2))
        q = fq * (c2 * C).sum(1)
        size = fq * (c2 * np.sqrt(c2)).sum()
        assert np.all(np.abs(f[6:9, k] - q) <= (eps + 12 * du / np.sqrt(c2.mean())) * size), (k, n)


@pytest.mark.parametrize("prec", ["FP64", "FP32"])
def test_a_cells_fields_do_not_depend_on_the_others(prec):
    """Dense on average (fewer cells per warp), sparse on average (the same
    cells ahead of 20,000 empty ones), and each cell alone."""
    cfg, pos, vel, cell = _flow(SIZES)
    f = _fields(cfg, pos, vel, prec)
    many = len(SIZES) + 20000
    g = _fields(dict(cfg, n=[many, 1, 1], hi=[float(many), 1.0, 1.0]), pos, vel, prec)
    assert np.array_equal(f, g[:, : len(SIZES)], equal_nan=True)
    one = dict(cfg, n=[1, 1, 1], hi=[1.0, 1.0, 1.0])
    for k, n in enumerate(SIZES):
        if n >= 2:
            h = _fields(one, pos[:, cell == k] - k, np.ascontiguousarray(vel[:, cell == k]), prec)
            assert np.array_equal(f[:, k], h[:, 0]), (k, n)


def test_time_of_a_dense_read():
    """One cell of 200,000 particles: the FP64 read (32 lanes, two passes of
    6250 rounds) against the FP32 one (16 lanes, 12500 rounds), which moves
    half the bytes: at most 3 times its time (four lanes took 6)."""
    import time

    import torch

    import paper_2506_23917_gb300 as sp

    cfg, pos, vel = W.homogeneous_box(200000, 1e-2, ppc=200000)
    t = []
    for prec in (sp.FP64, sp.FP32):
        s = sp.Sim(cfg, prec, capacity=200016)
        s.set_particles(0, pos, vel)
        s.moments(0, 0)
        reps = []
        for _ in range(10):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.moments(0, 0)
            reps.append(time.perf_counter() - t0)
        s.close()
        t.append(min(reps))
    assert t[0] < 3.0 * t[1], t
