"""Particles close enough to share nodes.  The step keeps one bit per node, and
the owner map only for particles whose circles came within reach of another's
(any other particle's nodes are its raster's row runs); these runs start with
gaps of 0.02 nodes and close them, so that particles overlap, in both team
sizes of the link kernel (few and many particles) and for windows of up to 64
columns.  Owner map, node flags and the index array's nodes against the
oracle's, node for node, after every step; a state saved among them continues
bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.oracle as orc  # noqa: E402
from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402


def flags_of(sim, nx, ny):
    pitch = (nx + 31) // 32 * 32
    buf = sim.get_state()
    off = 14 * ((pitch * ny + 63) // 64 * 64) * 4 + nx * ny * 4
    return buf[off:off + ny * pitch].reshape(ny, pitch)[:, :nx]


@pytest.mark.parametrize("shape,r,cols,rows", [
    ("disk", 6.4, 4, 3), ("disk", 6.4, 30, 20), ("ellipse", 7.7, 3, 3), ("ellipse", 5.2, 30, 17),
    ("disk", 28.4, 3, 1), ("ellipse", 28.4, 2, 2)])
def test_overlapping_particles(shape, r, cols, rows):
    rng = np.random.default_rng(int(10 * r) + cols)
    pitch = 2 * r + 0.02
    n = cols * rows
    parts = np.zeros(n, W.PARTICLE_DTYPE)
    k = np.arange(n)
    parts["x"], parts["y"] = r + 1.2 + pitch * (k % cols), r + 1.7 + pitch * (k // cols)
    parts["r"], parts["rho"], parts["T"] = r, 1.5, 1.0
    if shape == "ellipse":
        parts["b"], parts["theta"] = 0.9 * r, rng.uniform(-0.02, 0.02, n)  # tips face each other
        parts["omega"] = rng.normal(0, 2e-3, n)
    # the columns move towards each other in pairs (slowly: the fluid between
    # them has to leave)
    parts["ux"] = np.where(k % cols % 2, -0.02, 0.02)
    parts["uy"] = rng.uniform(-0.005, 0.005, n)
    nx, ny = int(pitch * cols + 14), int(pitch * rows + 11)
    prm = W.base_params(0.05, 0.71, 1e-6, eps_w=1e9)
    sim = lbm.Simulation(W.cavity(nx, ny), parts, prm)
    shared = 0
    for step in range(20):
        p0 = sim.particles()
        sim.step(1)
        p1 = sim.particles()
        o0, o1 = orc.raster(nx, ny, p0), orc.raster(nx, ny, p1)
        assert np.array_equal(sim.owner(), o1)
        exp = np.where(o1 >= 0, 1, np.where(o0 >= 0, 2, 0)).astype(np.uint8)
        assert np.array_equal(flags_of(sim, nx, ny), exp)
        node, _ = sim.slots()
        onode, _, over = orc.build_slots(nx, ny, o0, p0)
        assert over == 0 and np.array_equal(node, onode)
        assert sim.counters()[6] == (exp == 2).sum()
        alone = [orc.raster(nx, ny, p1[i:i + 1]) >= 0 for i in range(min(n, 40))]
        shared += int((np.sum(alone, 0) > 1).sum())
    assert shared > 0
    snap = sim.get_state()
    other = lbm.Simulation(W.cavity(nx, ny), parts, prm)
    other.set_state(snap)
    assert np.array_equal(other.get_state(), snap)
    for s in (sim, other):
        s.step(3)
    assert np.array_equal(sim.get_state(), other.get_state()) and np.array_equal(sim.owner(), other.owner())
    sim.close()
    other.close()


@pytest.mark.parametrize("n,periodic_x", [(0, 0), (40, 0), (40, 1)])
def test_sweeps_in_turn_equal_one_direction(n, periodic_x):
    """An FP32 lattice beyond L2 with few particles is swept up and down in
    turn; the same lattice in a batch always upwards.  Bit for bit."""
    nx, ny = 929, 1021
    rng = np.random.default_rng(n)
    lo = 9.0 + W.S_REP
    parts = W.rsa_disks(rng, n, 9.0, lo + 1, nx - lo - 2, lo, ny - lo - 1, min_gap=W.S_REP + 1.0) if n else None
    if n:
        parts["rho"], parts["T"] = 1.5, 1.0
        parts["ux"], parts["uy"] = rng.normal(0, 0.03, (2, n))
    dom = W.cavity(nx, ny, T_wall=(0.2, 0.9, 0.4, 0.0), periodic_x=periodic_x)
    sims = [lbm.Simulation(dom, parts, W.base_params(0.03, 0.71, 1e-4)) for _ in range(2)]
    b = lbm.Batch(sims[1:])
    for steps in (1, 12):
        sims[0].step(steps)
        b.step(steps)
        b.sync()
        assert np.array_equal(sims[0].get_state(), sims[1].get_state())
    b.close()
    for s in sims:
        s.close()
