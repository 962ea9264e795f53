"""Many particles with small zones: the link kernel's teams of one and two
warps per particle.  Against the oracle node for node (owner map, index array,
newborn count), and a batch, whose particles together take the small teams,
against its instances alone, whose own counts take four warps: bit for bit,
with particles apart and close enough to share nodes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.oracle as orc  # noqa: E402
from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402


def field(n, r, gap, shape="disk", seed=0):
    """n particles on a lattice, columns moving towards each other in pairs."""
    rng = np.random.default_rng(seed)
    c = int(np.ceil(np.sqrt(n)))
    k = np.arange(n)
    p = np.zeros(n, W.PARTICLE_DTYPE)
    p["x"], p["y"] = r + 1.2 + (2 * r + gap) * (k % c), r + 1.7 + (2 * r + gap) * (k // c)
    p["r"], p["rho"], p["T"] = r, 1.5, 1.0
    if shape == "ellipse":
        p["b"], p["theta"], p["omega"] = max(0.8 * r, 1.0), rng.uniform(-0.02, 0.02, n), rng.normal(0, 2e-3, n)
    p["ux"], p["uy"] = np.where(k % c % 2, -0.004, 0.004), rng.uniform(-0.002, 0.002, n)
    side = int((2 * r + gap) * c + 9)
    return side, p


def sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


# zones of 5 to 12 rows with more than 32 particles per SM, of 13 to 40 with
# more than 56
@pytest.mark.parametrize("shape,r,gap,per_sm", [
    ("disk", 1.0, 0.02, 33), ("disk", 1.0, 3.1, 33), ("disk", 2.3, 0.02, 33), ("ellipse", 3.0, 0.02, 33),
    ("disk", 4.5, 0.02, 33), ("disk", 4.51, 0.02, 57), ("ellipse", 6.2, 3.3, 57), ("disk", 18.5, 0.02, 57)])
def test_small_teams_match_the_oracle(shape, r, gap, per_sm):
    n = per_sm * sms() + 1
    side, p = field(n, r, gap, shape)
    sim = lbm.Simulation(W.cavity(side, side), p, W.base_params(0.05, 0.71, 1e-6, eps_w=1e9))
    for _ in range(3):
        p0 = sim.particles()
        o0 = orc.raster(side, side, p0)
        sim.step(1)
        o1 = orc.raster(side, side, sim.particles())
        assert np.array_equal(sim.owner(), o1)
        node, _ = sim.slots()
        onode, _, over = orc.build_slots(side, side, o0, p0)
        assert over == 0 and np.array_equal(node, onode)
        assert sim.counters()[6] == ((o0 >= 0) & (o1 < 0)).sum()
    sim.close()


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_BF16, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("shape,r,gap,per_sm", [
    ("disk", 1.0, 0.02, 40), ("ellipse", 2.4, 0.02, 40), ("disk", 4.5, 4.0, 40),
    ("disk", 5.0, 0.02, 60), ("ellipse", 8.3, 4.0, 60)])
def test_small_teams_equal_four_warps(shape, r, gap, per_sm, storage):
    prm = W.base_params(0.05, 0.71, 1e-6, eps_w=1e9)
    inst = [field(per_sm * sms() // 4, r, gap, shape, seed) for seed in range(4)]
    alone = []
    for side, p in inst:
        s = lbm.Simulation(W.cavity(side, side), p, prm, storage=storage)
        s.step(4)
        alone.append((s.get_state(), s.forces(), s.counters()))
        s.close()
    sims = [lbm.Simulation(W.cavity(side, side), p, prm, storage=storage) for side, p in inst]
    b = lbm.Batch(sims)
    b.step(4)
    b.sync()
    for s, (state, force, cnt) in zip(sims, alone):
        assert np.array_equal(s.get_state(), state) and np.array_equal(s.counters(), cnt)
        assert s.forces().tobytes() == force.tobytes()
    b.close()
    for s in sims:
        s.close()
