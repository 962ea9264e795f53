"""lbm_link_forces_noalloc takes its particles from device memory, where no host
code sees them.  One whose centre is not finite, or beyond any lattice, has no
links: planes and the other particles' forces are those of a call in which it
stands at (1e6, 1e6), on the row-mask path with windows of one and two words and
on the index-array path."""
import os
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_16597_gb300", "csrc")
BAD = [np.nan, np.inf, -np.inf, 1e300, 2.0 ** 31 - 20.0, -2.0 ** 31 + 3.0, 2.0 ** 31 - 60.5, 1e9]


def test_zone_origins_leave_room_for_every_offset():
    """Every zone origin is a clamped one: adding any window offset (two-node
    margin, a second word of 32 columns, zones of up to 712 nodes) stays within
    int32, as does the distance from the left end to the last column that lbm_init
    takes (nx ny < 2^31, ny >= 4); the right end lies beyond any lattice."""
    for name in os.listdir(CSRC):
        if name.endswith((".cu", ".cuh")):
            with open(os.path.join(CSRC, name)) as f:
                assert not re.search(r"[XY]0 = \(int\)floor", f.read()), name
    with open(os.path.join(CSRC, "lbm_internal.cuh")) as f:
        m = re.search(r"constexpr int kZoneLeft = -\(1 << (\d+)\), kZoneRight = 0x7fffffff - (\d+);", f.read())
    left, right = -(1 << int(m.group(1))), 2 ** 31 - 1 - int(m.group(2))
    assert right - 1 + 712 + 4 + 32 < 2 ** 31
    assert left - 1 - 4 > -2 ** 31 and (2 ** 31 - 1) // 4 - (left - 3) < 2 ** 31
    assert right > (2 ** 31 - 1) // 4


def call(A, ps, pitch, own, nx, ny, P, r_max):
    from paper_2308_16597_gb300 import lbm
    A = A.clone()
    o = torch.from_numpy(own).cuda()
    pd = torch.from_numpy(P.view(np.float64).reshape(-1, 10).copy()).cuda()
    F = torch.zeros((len(P), 3), dtype=torch.float64, device="cuda")
    lbm.lbm_link_forces_noalloc(A.data_ptr(), ps, pitch, o.data_ptr(), nx, ny, pd.data_ptr(), len(P), r_max, F.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return A.cpu().numpy(), F.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("axis", ["x", "y"])
@pytest.mark.parametrize("r,r_max", [(6.0, 6.0), (20.0, 20.0), (28.4, 28.5), (20.0, 40.0)])
def test_centres_outside_any_lattice_have_no_links(r, r_max, axis):
    from paper_2308_16597_gb300 import lbm
    nx, ny = 700, 515
    rng = np.random.default_rng(int(r) + int(r_max))
    n = 2 * len(BAD)
    P = np.zeros(n, lbm.PARTICLE_DTYPE)
    P["x"], P["y"] = rng.uniform(r + 40, nx - r - 3, n), rng.uniform(r + 40, ny - r - 3, n)
    P["r"], P["rho"], P["T"] = r, 1.5, 1.0
    P["ux"], P["uy"], P["omega"] = rng.normal(0, 5e-3, (3, n))
    j, i = np.mgrid[0:ny, 0:nx].astype(np.float64)
    own = np.full((ny, nx), -1, np.int32)
    for k in range(0, n, 2):  # the particles of odd index hold no node
        own[(i - P["x"][k]) ** 2 + (j - P["y"][k]) ** 2 <= r * r] = k
    pitch = 704
    ps = pitch * ny
    A = torch.from_numpy(rng.normal(0, 1e-3, (14, ps)).astype(np.float32)).cuda()
    P["x"][1::2], P["y"][1::2] = 1e6, 1e6
    a0, f0 = call(A, ps, pitch, own, nx, ny, P, r_max)
    P["x"][1::2], P["y"][1::2] = P["x"][::2], P["y"][::2]  # beside a particle but for the one coordinate
    P[axis][1::2] = BAD
    a1, f1 = call(A, ps, pitch, own, nx, ny, P, r_max)
    assert a0.tobytes() == a1.tobytes()
    assert f0[::2].tobytes() == f1[::2].tobytes() and (f0[::2] != 0).all()
