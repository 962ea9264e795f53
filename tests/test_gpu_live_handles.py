"""Handles alive side by side.  What a handle or batch prepares at its creation
(kernel shapes, shared memory) is its own: one created later, with smaller
zones and the same kernels, leaves the steps of the earlier one as they were,
launched directly, from graphs captured afterwards, and as a batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402

NX, NY = 600, 420


def disks(r, n):
    c = int((NX - 8) // (2 * r + 8))
    k = np.arange(n)
    p = np.zeros(n, W.PARTICLE_DTYPE)
    p["x"], p["y"] = r + 4.3 + (2 * r + 8) * (k % c), r + 4.6 + (2 * r + 8) * (k // c)
    p["r"], p["rho"], p["T"] = r, 1.5, 1.0
    return p


# (larger zones, smaller zones, particles): pairs whose zones take the same
# warps per particle
@pytest.mark.parametrize("big,small,n", [(28.4, 16.0, 2), (14.0, 5.0, 40)])
@pytest.mark.parametrize("storage", [lbm.LBM_STORE_FP32, lbm.LBM_STORE_BF16])
def test_a_later_handle_with_smaller_zones_changes_nothing(big, small, n, storage):
    dom, prm = W.cavity(NX, NY), W.base_params(0.05, 0.71, 1e-4)
    alone = lbm.Simulation(dom, disks(big, n), prm, storage=storage)
    alone.step(9)
    ref = alone.get_state()
    alone.close()
    for flags in (0, lbm.LBM_FLAG_NO_GRAPH):
        a = lbm.Simulation(dom, disks(big, n), prm, storage=storage, flags=flags)
        b = lbm.Simulation(dom, disks(small, n), prm, storage=storage, flags=flags)
        a.step(9)
        assert np.array_equal(a.get_state(), ref)
        b.step(9)
        b.sync()
        a.close()
        b.close()
    a = lbm.Simulation(dom, disks(big, n), prm, storage=storage)
    b = lbm.Simulation(dom, disks(small, n), prm, storage=storage)
    ba, bb = lbm.Batch([a]), lbm.Batch([b])
    ba.step(9)
    ba.sync()
    assert np.array_equal(a.get_state(), ref)
    for x in (ba, bb, a, b):
        x.close()
