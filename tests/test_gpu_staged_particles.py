"""The staged stream-collide of the 16-bit storages beside particles.  A single
lattice takes it from six row tiles per resident block on; the lattices here
are tall and narrow, with more than 6 x 16 row tiles per SM (no GPU holds more
than 16 blocks of 128 threads on one), so it runs whatever its occupancy.
Against the one-block-per-tile kernel, bit for bit: moving disks with newborn
nodes at tile edges, side walls, seams and the first and last rows; many
launches, replayed and direct; a batch of 1.5 million nodes or more; the fields
against the oracle; and the same cases in the bounds-checked build."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle.oracle as orc  # noqa: E402
from paper_2308_16597_gb300 import lbm, workloads as W  # noqa: E402

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
STORAGES = [lbm.LBM_STORE_BF16, lbm.LBM_STORE_FP16]
UNIT_ROUNDOFF = {lbm.LBM_STORE_BF16: 2.0 ** -8, lbm.LBM_STORE_FP16: 2.0 ** -11}


def tall():
    """Rows that make more than 6 tiles per block 16 blocks per SM would be."""
    return 6 * 16 * torch.cuda.get_device_properties(0).multi_processor_count + 5


def movers(nx, ny, per):
    """Moving disks at the side columns or seams, the first and last rows, the
    middle, and a touching pair."""
    r = min(6.0, nx / 8)
    edge = 2.2 if per else 1.0  # the clearance lbm_init asks for, or as far as they come in 26 steps
    x0, x1, xm = edge + r, nx - 1 - edge - r, 0.5 * nx
    P = [(x0, 40.3, -0.05, 0.03), (x1, 90.7, 0.05, 0.04), (xm, r + 0.9, 0.04, -0.04), (xm, ny - 1.9 - r, -0.04, 0.04),
         (xm, 0.5 * ny, 0.06, -0.05), (xm - r - 0.05, 0.7 * ny, 0.03, 0.01), (xm + r + 0.05, 0.7 * ny, -0.03, 0.02)]
    out = np.zeros(len(P), W.PARTICLE_DTYPE)
    for k, (x, y, ux, uy) in enumerate(P):
        out[k]["x"], out[k]["y"], out[k]["ux"], out[k]["uy"] = x, y, ux, uy
    if per:  # a seam turns a disk back no more than a wall does
        out["ux"][:2] *= -1
    out["r"], out["rho"], out["T"], out["omega"] = r, 2.0, 1.0, 2e-3
    return out


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("nx,per", [(64, 0), (70, 1), (200, 0), (257, 1), (300, 0)])
def test_staged_equals_unstaged_beside_moving_disks(nx, per, storage):
    ny = tall()
    dom = W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1), periodic_x=per)
    prm = W.base_params(0.05, 0.71, 1e-5, eps_w=1e6)
    a = lbm.Simulation(dom, movers(nx, ny, per), prm, storage=storage)
    b = lbm.Simulation(dom, movers(nx, ny, per), prm, storage=storage, flags=lbm.LBM_FLAG_SC_UNSTAGED)
    born = 0
    for n in (1, 2, 8, 15):
        a.step(n)
        b.step(n)
        assert np.array_equal(a.get_state(), b.get_state())
        assert np.array_equal(a.counters(), b.counters())
        born += int(a.counters()[6])
    assert born > 0
    a.close()
    b.close()


@pytest.mark.parametrize("storage", STORAGES)
def test_staged_fields_match_the_oracle(storage):
    nx, ny = 64, tall()
    dom = W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1))
    prm = W.base_params(0.05, 0.71, 1e-5, eps_w=1e6)
    sim, ref = lbm.Simulation(dom, movers(nx, ny, 0), prm, storage=storage), orc.Oracle(dom, movers(nx, ny, 0), prm)
    sim.step(6)
    assert ref.step(6) == 0
    got, exp = sim.fields(), ref.fields()
    fluid = ~np.isnan(exp[0]) & ~np.isnan(got[0])
    for name, x, y in zip(("rho-1", "ux", "uy", "T"), got, exp):
        x, y = x[fluid].astype(np.float64), y[fluid] - (1.0 if name == "rho-1" else 0.0)
        assert np.linalg.norm(x - y) <= 5.0 * UNIT_ROUNDOFF[storage] * np.linalg.norm(y), name
    sim.close()


@pytest.mark.parametrize("nx,times", [(33, 1), (500, 1), (500, 3)])  # claims of 1, 2 and 4 tiles with 8 blocks per SM
def test_work_counter_is_reset_between_launches(nx, times):
    dom, prm = W.cavity(nx, times * tall(), T_wall=(0.0, 0.0, 1.0, 0.0)), W.base_params(0.05, 0.71, 1e-4)
    sims = [lbm.Simulation(dom, None, prm, storage=lbm.LBM_STORE_BF16, flags=f)
            for f in (0, lbm.LBM_FLAG_SC_UNSTAGED, lbm.LBM_FLAG_NO_GRAPH)]
    for n in (1, 2, 9, 16):
        for s in sims:
            s.step(n)
    states = [s.get_state() for s in sims]
    assert np.array_equal(states[0], states[1]) and np.array_equal(states[0], states[2])
    for s in sims:
        s.close()


@pytest.mark.parametrize("storage", STORAGES)
def test_staged_batch_equals_each_instance_alone_beside_moving_disks(storage):
    """Instances on either side of the sizes that take the staged kernel alone,
    one of them an odd step ahead."""
    prm = W.base_params(0.05, 0.71, 1e-5, eps_w=1e6)
    shapes = [(70, 300, 1), (257, 181, 0), (64, 400, 0), (1300, 1300, 0)]  # 1.7 million nodes and more: staged
    def make():
        out = [lbm.Simulation(W.cavity(nx, ny, T_wall=(0.3, 0.8, 1.0, 0.1), periodic_x=per), movers(nx, ny, per), prm,
                              storage=storage) for nx, ny, per in shapes]
        out[1].step(3)
        out[1].sync()
        return out
    sims, alone = make(), make()
    b = lbm.Batch(sims)
    born = 0
    for n in (1, 2, 13):
        b.step(n)
        b.sync()
        for s, a in zip(sims, alone):
            a.step(n)
            assert np.array_equal(s.get_state(), a.get_state())
            assert np.array_equal(s.counters(), a.counters())
            born += int(s.counters()[6])
    assert born > 0
    b.close()
    for s in sims + alone:
        s.close()


CHILD = textwrap.dedent(r"""
    import numpy as np
    from paper_2308_16597_gb300 import lbm, workloads as W
    from tests.test_gpu_staged_particles import STORAGES, movers, tall

    prm = W.base_params(0.05, 0.71, 1e-5, eps_w=1e6)
    for storage in STORAGES:
        for nx, px, py in ((64, 0, 0), (257, 1, 0), (300, 0, 0), (40, 0, 1)):
            ny = tall()
            s = lbm.Simulation(W.cavity(nx, ny, periodic_x=px, periodic_y=py), movers(nx, ny, px) if not py else None,
                               prm, storage=storage)
            s.step(9)
            s.sync()                    # raises on LBM_EBOUNDS
            s.set_state(s.get_state())  # the bits of a restored image
            s.step(2)
            s.sync()
            s.close()
        sims = [lbm.Simulation(W.cavity(nx, ny), movers(nx, ny, 0), prm, storage=storage)
                for nx, ny in ((70, 300), (257, 181), (1300, 1300))]
        b = lbm.Batch(sims)
        b.step(9)
        b.sync()
        b.close()
        for s in sims:
            s.close()
    print("checked build: no out-of-bounds index")
""")


def test_bounds_checked_build_runs_the_staged_kernel(tmp_path):
    from paper_2308_16597_gb300 import build as B
    lib = B.build(force=True, extra=["-DLBM_CHECK"], out=str(tmp_path))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, LBM_LIBRARY=lib, PYTHONPATH=ROOT),
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "no out-of-bounds index" in r.stdout
