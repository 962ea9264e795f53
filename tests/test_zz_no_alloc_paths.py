"""The two paths of lbm_link_forces_noalloc: zones of at most 60 nodes a side
(chosen by r_max) take the row-mask kernels, larger ones the index array in
memory.  The same particles passed with a small and a large r_max go through
one and the other; planes and forces must agree bit for bit (the per-link
arithmetic is shared and the sums are exact integers)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2308_16597_gb300 import lbm  # noqa: E402


def owner_map(nx, ny, parts):
    own = np.full((ny, nx), -1, np.int32)
    j, i = np.mgrid[0:ny, 0:nx].astype(np.float64)
    for k, p in enumerate(parts):
        dx, dy = i - p["x"], j - p["y"]
        c, s = np.cos(p["theta"]), np.sin(p["theta"])
        b = p["b"] if p["b"] > 0 else p["r"]
        u, v = dx * c + dy * s, dy * c - dx * s
        own[(u / p["r"]) ** 2 + (v / b) ** 2 <= 1.0] = k
    return own


def particles(nx, ny, radii, shape, rng):
    n = len(radii)
    P = np.zeros(n, lbm.PARTICLE_DTYPE)
    # overlaps and particles over the edge are allowed: the owner map decides
    P["x"], P["y"] = rng.uniform(0, nx, n), rng.uniform(0, ny, n)
    P["r"] = radii
    if shape == "ellipse":
        P["b"] = np.maximum(0.5 * P["r"], 1.0)
        P["theta"] = rng.uniform(-4.0, 4.0, n)
    P["ux"], P["uy"], P["omega"] = rng.normal(0, 5e-3, (3, n))
    P["rho"], P["T"] = 1.5, rng.uniform(0.5, 1.0, n)
    return P


def call(A, ps, pitch, own, nx, ny, P, r_max):
    n = len(P)
    A = A.clone()
    o = torch.from_numpy(own).cuda()
    pd = torch.from_numpy(P.view(np.float64).reshape(-1, 10).copy()).cuda()
    F = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    lbm.lbm_link_forces_noalloc(A.data_ptr(), ps, pitch, o.data_ptr(), nx, ny, pd.data_ptr(), n, r_max, F.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return A.cpu().numpy(), F.cpu().numpy()


@pytest.mark.parametrize("shape", ["disk", "ellipse"])
@pytest.mark.parametrize("nx,ny,radii", [
    (64, 48, [6.0, 1.0]),                 # the smallest radius
    (257, 130, [10.0] * 9),               # overlapping: lines with two links
    (333, 301, [14.2, 28.4, 28.5, 3.7]),  # windows of 33 to 64 columns
    (700, 515, list(np.linspace(2.0, 28.0, 129)))])
def test_row_mask_path_equals_the_index_array_path(shape, nx, ny, radii):
    rng = np.random.default_rng(nx)
    P = particles(nx, ny, np.array(radii), shape, rng)
    own = owner_map(nx, ny, P)
    own[::17, ::13] = -1  # holes: lines crossing the owner more than once
    pitch = (nx + 31) // 32 * 32
    ps = (pitch * ny + 63) // 64 * 64
    A = torch.from_numpy(rng.normal(0, 1e-3, (14, ps)).astype(np.float32)).cuda()
    a0, f0 = call(A, ps, pitch, own, nx, ny, P, 28.5)
    a1, f1 = call(A, ps, pitch, own, nx, ny, P, 40.0)
    assert a0.tobytes() == a1.tobytes()
    assert np.array_equal(f0, f1, equal_nan=True)
    assert (a0 != A.cpu().numpy()).any()
    # one particle that breaks the rule: no plane written, every force NaN
    P["r"][0] = 0.5
    a2, f2 = call(A, ps, pitch, own, nx, ny, P, 28.5)
    assert a2.tobytes() == A.cpu().numpy().tobytes() and np.isnan(f2).all()


def test_call_can_be_captured_and_replayed():
    """The row-mask path's two launches (the second one ahead of the first
    one's end) in a captured graph, replayed on restored planes."""
    nx, ny = 257, 130
    rng = np.random.default_rng(3)
    P = particles(nx, ny, np.array([10.0] * 5), "disk", rng)
    own = owner_map(nx, ny, P)
    pitch, ps = 288, 288 * ny
    A = torch.from_numpy(rng.normal(0, 1e-3, (14, ps)).astype(np.float32)).cuda()
    a0, f0 = call(A, ps, pitch, own, nx, ny, P, 10.0)
    o = torch.from_numpy(own).cuda()
    pd = torch.from_numpy(P.view(np.float64).reshape(-1, 10).copy()).cuda()
    B, F = A.clone(), torch.zeros((len(P), 3), dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        lbm.lbm_link_forces_noalloc(B.data_ptr(), ps, pitch, o.data_ptr(), nx, ny, pd.data_ptr(), len(P), 10.0,
                                    F.data_ptr(), torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        B.copy_(A)
        F.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert B.cpu().numpy().tobytes() == a0.tobytes() and F.cpu().numpy().tobytes() == f0.tobytes()
