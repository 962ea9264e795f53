"""lbm_get_owner and lbm_get_state only read.  They spell the maps of a state
out of the node bits, the row runs and the owner map of the crowded particles;
nothing of the handle's workspace changes, whatever the step's parity, so a
batch whose steps are still in flight is not disturbed either.  A restored
image's own owner map comes back, with the particles' nodes over it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.oracle as orc  # noqa: E402
from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402

NX, NY = 203, 161
OWN = slice(14 * ((224 * NY + 63) // 64 * 64) * 4, 14 * ((224 * NY + 63) // 64 * 64) * 4 + 4 * NX * NY)


def start(n, storage=lbm.LBM_STORE_FP32):
    p = np.zeros(n, W.PARTICLE_DTYPE)
    # two touching disks (crowded), one alone, one at the walls
    p["x"], p["y"] = [60.2, 88.2, 150.6, 14.0][:n], [80.0, 80.3, 100.4, 14.5][:n]
    p["r"], p["rho"], p["T"] = 14.0, 1.5, 1.0
    p["ux"] = [0.02, -0.02, 0.03, 0.0][:n]
    return lbm.Simulation(W.cavity(NX, NY), p, W.base_params(0.05, 0.71, 1e-5, eps_w=1e6), storage=storage)


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("n", [0, 4])
def test_inspection_leaves_the_workspace_alone(n, storage):
    sim = start(n, storage)
    for steps in (0, 1, 4, 3):
        sim.step(steps)
        sim.sync()
        before = sim.workspace.clone()
        own, image = sim.owner(), sim.get_state()
        assert torch.equal(sim.workspace, before)
        assert np.array_equal(own, orc.raster(NX, NY, sim.particles()))
        if storage == lbm.LBM_STORE_FP32:
            assert np.array_equal(image[OWN].view(np.int32).reshape(NY, NX), own)
    sim.close()


def test_an_images_owner_map_comes_back():
    sim = start(4)
    sim.step(5)
    image = sim.get_state()
    own = image[OWN].view(np.int32).reshape(NY, NX)
    full = own.copy()
    own[3, 199], full[3, 199] = 2, 2  # a fluid node that the image gives to a particle
    own[80, 60] = -1                  # one inside a particle: the raster goes over the image
    sim.set_state(image)
    assert np.array_equal(sim.owner(), full)
    assert np.array_equal(sim.get_state()[OWN].view(np.int32).reshape(NY, NX), full)
    # an image of any alignment in host memory
    raw = np.zeros(image.size + 1, np.uint8)
    lbm._check(lbm.library().lbm_get_state(sim.h, raw[1:].ctypes.data, image.size), "lbm_get_state")
    assert np.array_equal(raw[1:], sim.get_state())
    sim.close()
