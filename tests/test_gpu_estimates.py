"""Decisions that an FP32 estimate may settle ahead of the FP64 arithmetic, at
the lines where the estimate must hand over: cells of coordinates next to cell
faces, flights that graze a body or end next to a wall, candidate counts next
to whole numbers, splits next to pure DSMC.  (NTC and Shakhov decisions: the
full-size steps against the oracle draw millions of them.)"""
import numpy as np
import pytest

import oracle
from paper_2506_23917_gb300 import workloads as W
from tests.test_gpu_parity import compare_state, compare_surface

pytestmark = pytest.mark.gpu
SHIFTS = [(1.0, 0.0), (1e-6, 0.0), (1.0, 1000.0), (1e3, -5e7), (1e-9, 1.0)]  # length scale, offset of the box
REL = [0.0, 1e-15, 1e-12, 1e-9, 1e-8, 1e-7, 3e-7, 1e-6, 3e-6, 1e-5, 1e-4]


def _quiet(cfg, **kw):
    """No collisions: the gas holds next to no molecules, and no draw rounds its count up."""
    return dict(cfg, mode=W.MODE_DSMC, Fn=1e-300, cell_volume=None, n_steady=0, **kw)


@pytest.mark.parametrize("scale,shift", SHIFTS)
@pytest.mark.parametrize("n", [[7], [1000], [131071], [40, 25], [9, 8, 7]])
def test_cells_of_coordinates_at_faces(n, scale, shift):
    import paper_2506_23917_gb300 as sp

    rng = np.random.Generator(np.random.PCG64(8))
    dim = len(n)
    lo = [shift + scale * a for a in (0.25, -0.4, -0.1)[:dim]]
    hi = [a + scale * b for a, b in zip(lo, (1.0, 1.7, 0.3))]
    cfg = _quiet(W.base_config(dim, n, lo, hi), dt_fixed=1e-3)
    m = 60000
    x = np.empty((dim, m))
    for d in range(dim):
        face = lo[d] + rng.integers(0, n[d] + 1, m) * ((hi[d] - lo[d]) / n[d])
        off = rng.choice(REL, m) * rng.choice([-1, 1], m) * (hi[d] - lo[d] + abs(lo[d]) * rng.integers(0, 2, m))
        x[d] = np.clip(np.nextafter(face + off, face + rng.choice([-1.0, 1.0], m) * 1e300), lo[d], hi[d])
    cell = np.zeros(m, dtype=np.int64)
    for d in reversed(range(dim)):
        i = np.floor((x[d] - lo[d]) * (n[d] / (hi[d] - lo[d])))
        cell = np.clip(i, 0, n[d] - 1).astype(np.int64) + n[d] * cell
    s = sp.Sim(cfg, sp.FP64, capacity=m)
    s.set_particles(0, x, rng.normal(0, 1, (3, m)))
    p, _, c = s.particles(0)
    s.close()
    order = np.argsort(cell, kind="stable")
    assert np.array_equal(c, cell[order])
    assert np.array_equal(p, x[:, order])


def _flights(rng, lo, hi, c, r, dt, n):
    """Flights of time dt that pass a body (circle or sphere of radius r about
    c) along a tangent, end next to it, or end next to a face of the box."""
    dim = len(lo)
    span = min(hi - lo)
    X, V = [], []

    def unit():
        u = rng.normal(0, 1, dim)
        return u / np.linalg.norm(u)

    while len(X) < n:
        rel = rng.choice(REL) * rng.choice([-1, 1])
        kind = rng.integers(0, 3)
        if kind == 2:  # ends next to a face
            d, side = rng.integers(0, dim), rng.integers(0, 2)
            e = lo + rng.random(dim) * (hi - lo)
            e[d] = (hi[d] if side else lo[d]) + rel * rng.choice([span, abs(lo[d]) + abs(hi[d])])
            v = unit() * span * rng.uniform(0.05, 0.4) / dt
            x = e - v * dt
        else:
            u = unit()
            at = c + r * (1.0 + rel) * u
            v = unit() * span * rng.uniform(0.05, 0.4) / dt
            if kind == 0:  # along the tangent
                v -= (v @ u) * u
                x = at - v * dt * rng.choice([rng.uniform(0.01, 0.99), 1.0, 1.0 - 1e-7, 1e-7])
            else:  # ends next to the body
                x = at - v * dt
        if np.all(x > lo) and np.all(x < hi) and np.linalg.norm(x - c) > r * (1 + 1e-12):
            X.append(x)
            V.append(np.concatenate([v, rng.normal(0, 1, 3 - dim)]))
    return np.array(X).T, np.array(V).T


@pytest.mark.parametrize("scale,shift", SHIFTS[:4])
@pytest.mark.parametrize("dim", [2, 3])
def test_flights_that_graze(dim, scale, shift):
    import paper_2506_23917_gb300 as sp

    cfg = (W.box2d(inflow=False) if dim == 2 else W.box3d())[0]
    cfg = _quiet(cfg, dt_fixed=0.05, n_surf=40, seed=9)
    cfg["face_bc"] = [W.BC_DIFFUSE, W.BC_OUTFLOW, W.BC_SPECULAR, W.BC_DIFFUSE, W.BC_SPECULAR, W.BC_SPECULAR]
    for k in ("lo", "hi", "body_c"):
        cfg[k] = [scale * a + (shift if d < dim else 0.0) for d, a in enumerate(cfg[k])]
    cfg["body_r"] *= scale
    cfg["face_T"] = [scale * scale] * 6
    cfg["body_Tw"] = scale * scale
    rng = np.random.Generator(np.random.PCG64(12))
    lo, hi, c = (np.array(cfg[k][:dim]) for k in ("lo", "hi", "body_c"))
    pos, vel = _flights(rng, lo, hi, c, cfg["body_r"], 0.05, 20000)
    o = oracle.Oracle(cfg)
    o.set_particles(pos, vel)
    s = sp.Sim(cfg, sp.FP64, capacity=30000)
    s.set_particles(0, pos, vel)
    compare_state(o, s, what="before")
    o.step(1)
    s.step(1)
    compare_state(o, s, what="after")
    compare_surface(o, s, what="hits")
    assert o.M < pos.shape[1]  # (some left through the outflow face)
    s.close()


def test_candidate_counts_next_to_whole_numbers():
    """FP32 state, FP64 cells, DSMC forced: N_col = floor(N (N - 1) F_N
    (sigma c)_max dt / (2 V) + u) of every cell, formed here in 64 bits."""
    import paper_2506_23917_gb300 as sp

    rng = np.random.Generator(np.random.PCG64(4))
    nc = 30000
    n = rng.integers(2, 40, nc)
    cfg = dict(W.sod(ncell=nc, n_steady=0)[0], mode=W.MODE_DSMC, seed=77)
    cell = np.repeat(np.arange(nc), n)
    pos = ((cell + rng.uniform(0.05, 0.95, len(cell))) / nc)[None].astype(np.float32).astype(np.float64)
    vel = rng.normal(0, 1, (3, len(cell))).astype(np.float32).astype(np.float64)
    # about 20 candidates in a cell of 20
    cfg["Fn"] *= 5e3
    s = sp.Sim(cfg, sp.FP32, capacity=len(cell) + 64)
    s.set_particles(0, pos, vel)
    s.set_record(True)
    dt, smax, N = s.dt(0), s.sigc_max(0).astype(np.float32).astype(np.float64), np.diff(s.cell_start(0)).astype(float)
    s.step(1)
    got = s.record(0)[0][0]
    assert abs(s.dt(0) / dt - 1) < 1e-12  # (the least dt_c, of the same state, is not lost)
    s.close()
    u = np.array([(2 * (int(oracle.philox([0, k, 0xFFFFFFFF, 1 << 24], [77, 0])[0]) >> 9) + 1) * 2.0**-24
                  for k in range(nc)])
    x = 0.5 * N * (N - 1) * cfg["Fn"] * smax * dt * nc + u
    assert np.array_equal(got, np.floor(x).astype(np.int64))
    near = np.abs(x - np.round(x)) < 2e-4 * x
    assert near.sum() > 50 and 2 < np.median(x) < 2000, (near.sum(), np.median(x))


@pytest.mark.parametrize("lam", [2e-5, 2e-4, 2.2e-4])
def test_which_cells_are_pure_dsmc(lam):
    """FP32 state, FP64 cells: a step samples a split ratio of exactly 1 in the
    cells with tau >= dt_c and less in the others, tau and dt_c formed here in
    64 bits from the FP32 particles.  The step's |C|^2 are FP32: two roundings
    of C count twice, three more follow, so T errs by up to 7 x 2^-24 and
    tau / dt_c, which goes with T to a power of at most 1, by less than 1e-6."""
    import paper_2506_23917_gb300 as sp

    cfg, regions = W.sod(ncell=4000, ppc_left=60.0, lam_left=lam, n_steady=0)
    pos, vel = (a.astype(np.float32).astype(np.float64) for a in W.fill_regions(cfg, regions, 3))
    s = sp.Sim(cfg, sp.FP32, capacity=vel.shape[1] + 64)
    s.set_particles(0, pos, vel)
    start = s.cell_start(0).astype(np.int64)
    v = s.particles(0)[1]
    s.step(1)
    got = s.moments(0, 1)[11]
    s.close()
    x = np.full(4000, np.inf)
    for k in range(4000):
        c = v[:, start[k]:start[k + 1]]
        n = c.shape[1]
        if n < 2:
            continue
        u = c.mean(1)
        T = ((c - u[:, None]) ** 2).sum() / (3 * cfg["R"] * (n - 1))
        dens = n * cfg["Fn"] * 4000
        tau = cfg["mu_ref"] * (T / cfg["T_ref"]) ** cfg["omega"] / (dens * cfg["m"] * cfg["R"] * T)
        x[k] = tau * (np.sqrt(u @ u) + np.sqrt(cfg["gamma"] * cfg["R"] * T)) * 4000
    assert np.all(got[x > 1 + 1e-6] == 1.0)
    assert np.all(got[x < 1 - 1e-6] < 1.0)
    assert np.sum(np.abs(x - 1) < 0.03) > 40  # (cells next to the line)
