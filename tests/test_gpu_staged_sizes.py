"""The staged stream-collide where the library chooses it: a single 16-bit
lattice of 6 row tiles or more per resident block, and batches.  Against the
one-block-per-tile kernel, bit for bit, with tile counts around the chunk
rule's lines (claims of 1, 2 and 4 tiles; the last claims past the end), ragged
widths, and small lattices beside a large one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
W5 = np.array([0.6] + [0.1] * 4)


def start(dom, nx, ny, storage, flags):
    s = lbm.Simulation(dom, None, W.base_params(0.03, 0.71, 3e-3), storage=storage, flags=flags)
    f, g = W.random_state(nx, ny, 5, W9, W5, amp=1e-2)
    s.set_distributions(f, g)
    return s


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_BF16, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("nx,ny,per", [(300, 3700, (0, 0)), (257, 4001, (1, 0)), (40, 19500, (0, 1)),
                                       (250, 38950, (0, 0))])
def test_large_lattices_equal_the_unstaged_kernel(nx, ny, per, storage):
    dom = W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1), periodic_x=per[0], periodic_y=per[1])
    a, b = start(dom, nx, ny, storage, 0), start(dom, nx, ny, storage, lbm.LBM_FLAG_SC_UNSTAGED)
    for n in (1, 4):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


@pytest.mark.parametrize("storage", [lbm.LBM_STORE_BF16, lbm.LBM_STORE_FP16])
@pytest.mark.parametrize("nx,ny", [(4, 4), (70, 50), (257, 33), (300, 1301)])
def test_small_lattices_in_a_staged_batch_equal_themselves_alone(nx, ny, storage):
    dom, big = W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1)), W.cavity(1300, 1200)
    a, b = start(dom, nx, ny, storage, 0), start(dom, nx, ny, storage, 0)
    c = lbm.Simulation(big, None, W.base_params(0.03, 0.71, 0.0), storage=storage)
    bt = lbm.Batch([a, c])  # large enough for the staged kernel
    bt.step(5)
    bt.sync()
    b.step(5)
    assert np.array_equal(a.get_state(), b.get_state())
    bt.close()
    for s in (a, b, c):
        s.close()
