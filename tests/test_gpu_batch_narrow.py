"""A batch of narrow FP32 lattices takes tiles of several rows from its creation
on; one with a wider lattice among them takes one row a tile.  Either gives the
states of its instances alone, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
W5 = np.array([0.6] + [0.1] * 4)


def start(nx, ny, k):
    parts = np.zeros(1, W.PARTICLE_DTYPE)
    parts["x"], parts["y"], parts["r"], parts["rho"], parts["T"] = nx / 2 - 0.3, ny / 2 + 0.2, 4.0, 1.5, 1.0
    dom = W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1), periodic_y=k % 2)
    s = lbm.Simulation(dom, parts if min(nx, ny) >= 20 else None, W.base_params(0.03, 0.71, 1e-4))
    s.set_distributions(*W.random_state(nx, ny, 5 + k, W9, W5, amp=1e-2))
    return s


@pytest.mark.parametrize("sizes", [
    [(4, 4), (20, 301), (32, 50), (33, 7), (64, 130)],  # at most 64 nodes a row: 32 x 4 threads
    [(20, 301), (65, 40)]])
def test_narrow_batch_equals_each_instance_alone(sizes):
    sims = [start(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    alone = [start(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    b = lbm.Batch(sims)
    for steps in (1, 6):
        b.step(steps)
        b.sync()
        for s, a in zip(sims, alone):
            a.step(steps)
            assert np.array_equal(s.get_state(), a.get_state())
    b.close()
    for s in sims + alone:
        s.close()
