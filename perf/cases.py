"""The work a user of this library has it do, as cases that can be timed.

Every case goes through the public binding (``paper_2308_16597_gb300.lbm``):
a ``Simulation`` advanced some steps and read back, a ``Batch`` of independent
simulations, a ``Server`` that takes requests from submission to result, and
the allocation-free link forces.  Sizes are those of this repository's own
workloads, tests and benchmark.

A pass of a simulation enqueues its steps, the macroscopic fields on the
device and the particle states into page-locked memory, and waits for nothing
(a batch synchronises before its instances are read, as its contract asks; a
server call returns host arrays).

``exact`` restates the method in FP64 with plain torch operations: D2Q9 MRT
flow and D2Q5 MRT temperature, half-way walls, curved bounce-back with
momentum exchange, Newton-Euler particles with spring repulsion, refilling.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_16597_gb300 import lbm

STORAGE = {"fp32": lbm.LBM_STORE_FP32, "bf16": lbm.LBM_STORE_BF16, "fp16": lbm.LBM_STORE_FP16}
S_REP = 3.0  # repulsion range, lattice units


def _sim(name, nx, ny, n, storage, steps, shape="disk", r_lo=10.0, r_hi=10.0, y_lo=0.5, setup="settle", nu=0.02,
         pr=0.71, u_ff=0.03, spin=16):
    """A simulation case: n particles of semi-major axis r_lo..r_hi (ellipses: aspect ratio 2) with centres above
    y_lo ny; setup "settle" (hot particles sink in a cold closed cavity), "bed" (a force drives the fluid through
    fixed particles, periodic in x), "heated" (no particles, the left wall hot) or "lattice" (settle, with the
    particles on a square lattice of pitch 50).  u_ff: free-fall velocity sqrt(g beta dT H); spin: steps taken from
    rest before the first pass (a program is rarely at its first step)."""
    return dict(name=name, kind="sim", nx=nx, ny=ny, n=n, storage=storage, steps=steps, shape=shape, r_lo=r_lo,
                r_hi=r_hi, y_lo=y_lo, setup=setup, nu=nu, pr=pr, u_ff=u_ff, spin=spin)


def listed():
    return [
        # the smallest call: one step of two hot disks, everything read back (a coupling or a viewer asks for every
        # step; the smoke run's size)
        _sim("tiny_64x48", 64, 48, 2, "fp32", 1, r_lo=6.0, r_hi=6.0, nu=0.05),
        # a validation-size run: the parity cavity, latency of the step's launches
        _sim("cavity_256_8disks", 256, 256, 8, "fp32", 20),
        # the same size with spinning ellipses in BF16 storage
        _sim("cavity_256_6ellipses_bf16", 256, 256, 6, "bf16", 20, shape="ellipse", r_lo=12.0, r_hi=12.0),
        # natural convection without particles on a ragged lattice: stream-collide alone
        _sim("heated_777x513", 777, 513, 0, "fp32", 20, setup="heated"),
        # flow through a bed of fixed disks of several sizes, periodic in x, odd sizes, FP16 storage
        _sim("bed_1531x1021_fp16", 1531, 1021, 300, "fp16", 20, r_lo=4.0, r_hi=14.0, y_lo=0.1, setup="bed"),
        # the paper's elliptical particles (Sec. 2.6.3): 129 ellipses 50 x 25 in 1000 x 2000
        _sim("ellipses_1000x2000", 1000, 2000, 129, "fp32", 20, shape="ellipse", r_lo=25.0, r_hi=25.0, nu=0.01,
             pr=5.0),
        # the benchmark: 4000^2, 4800 hot disks, FP32 and reduced storage
        _sim("sedimentation_4000", 4000, 4000, 4800, "fp32", 20, y_lo=0.4, u_ff=0.0596),
        _sim("sedimentation_4000_bf16", 4000, 4000, 4800, "bf16", 20, y_lo=0.4, u_ff=0.0596),
        # the paper's own 4800-particle benchmark: d = 40 on a lattice of pitch 50, 38 % solid
        _sim("paper_4800_d40_fp16", 4000, 4000, 4800, "fp16", 20, r_lo=20.0, r_hi=20.0, y_lo=0.25, setup="lattice",
             nu=0.01, pr=5.0, u_ff=0.0194),
        # a parameter study: 64 cavities of 256..1024 a side stepped as one batch
        dict(name="ensemble_64", kind="batch", count=64, lo=256, hi=1024, r_lo=6.0, r_hi=12.0, fill=0.2,
             storage="fp32", steps=20),
        # forces for a caller that owns its buffers and cannot allocate: 1200 disks in 2000^2
        dict(name="link_forces_2000", kind="forces", nx=2000, ny=2000, n=1200, shape="disk", r_lo=10.0, r_hi=10.0),
        # serving: requests of several sizes from submission to results in host memory
        dict(name="served_5_bf16", kind="serve", count=5, lo=512, hi=1024, r_lo=10.0, r_hi=10.0, fill=0.2,
             storage="bf16", steps=96, tick=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of these ranges: mostly single simulations, any storage, sides from 48 to 4000."""
    kind = rng.choice(("sim", "sim", "sim", "sim", "sim", "batch", "forces", "serve"))
    storage = rng.choice(tuple(STORAGE))
    if kind == "batch":
        lo = _log_int(rng, 64, 300)
        return dict(kind="batch", count=_log_int(rng, 2, 48), lo=lo, hi=_log_int(rng, lo, 1000), r_lo=5.0,
                    r_hi=rng.uniform(6.0, 12.0), fill=rng.uniform(0.05, 0.2), storage=storage,
                    steps=rng.randint(4, 20))
    if kind == "serve":
        lo = _log_int(rng, 128, 700)
        return dict(kind="serve", count=rng.randint(2, 5), lo=lo, hi=_log_int(rng, lo, 1000), r_lo=8.0,
                    r_hi=rng.uniform(8.0, 12.0), fill=rng.uniform(0.05, 0.2), storage=storage,
                    steps=rng.randint(20, 90), tick=rng.randint(8, 40))
    nx, ny = _log_int(rng, 64, 3900), _log_int(rng, 64, 3900)
    shape = rng.choice(("disk", "disk", "ellipse"))
    cap = min(27.0, min(nx, ny) / 8.0)
    r_lo = rng.uniform(min(5.0, cap), cap)
    r_hi = rng.uniform(r_lo, cap)
    y_lo = rng.uniform(0.1, 0.5)
    room = (nx - 2 * r_hi - 8) * ((1 - y_lo) * ny - 2 * r_hi - 8)
    n = int(max(1, min(4800, rng.uniform(0.02, 0.18) * room / (math.pi * r_hi ** 2))))
    if kind == "forces":
        n = min(n, 2097152 // (12 * (math.ceil(2 * r_hi) + 3)))
        return dict(kind="forces", nx=nx, ny=ny, n=n, shape=shape, r_lo=r_lo, r_hi=r_hi)
    setup = rng.choice(("settle", "settle", "settle", "bed", "heated"))
    if setup == "heated":
        n = 0
    if setup == "bed" and storage == "bf16":
        storage = "fp16"  # 8 bits do not resolve the density of so slow a flow
    case = _sim("", nx, ny, n, storage, rng.choice((1, 2, 5, 8, 13, 20)), shape=shape, r_lo=r_lo, r_hi=r_hi, y_lo=y_lo,
                setup=setup, nu=rng.uniform(0.02, 0.06), pr=rng.uniform(0.7, 2.0), u_ff=rng.uniform(0.01, 0.04))
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _place(rng, n, radii, xlo, xhi, ylo, yhi, gap):
    """Random sequential addition of n particles whose circumscribed circles keep `gap` apart."""
    cell = 2.0 * float(radii.max()) + gap
    grid, xs, ys = {}, [], []
    for x, y in zip(rng.uniform(xlo, xhi, 40 * n + 40).tolist(), rng.uniform(ylo, yhi, 40 * n + 40).tolist()):
        if len(xs) == n:
            break
        r, cx, cy = float(radii[len(xs)]), int(x // cell), int(y // cell)
        near = (k for gx in (cx - 1, cx, cx + 1) for gy in (cy - 1, cy, cy + 1) for k in grid.get((gx, gy), ()))
        if all((x - xs[k]) ** 2 + (y - ys[k]) ** 2 >= (r + radii[k] + gap) ** 2 for k in near):
            grid.setdefault((cx, cy), []).append(len(xs))
            xs.append(x)
            ys.append(y)
    if len(xs) < n:
        raise RuntimeError("%d particles do not fit" % n)
    return np.array(xs), np.array(ys)


def _particles(rng, nx, ny, n, shape, r_lo, r_hi, y_lo, setup):
    if n == 0:
        return np.zeros(0, lbm.PARTICLE_DTYPE)
    radii = rng.uniform(r_lo, r_hi, n) if r_hi > r_lo else np.full(n, r_lo)
    radii[0] = r_hi
    if setup == "lattice":
        per = nx // 50
        k = np.arange(n)
        x = 25.0 + 50.0 * (k % per) + rng.uniform(-1.5, 1.5, n)
        y = ny - 25.0 - 50.0 * (k // per) + rng.uniform(-1.5, 1.5, n)
    else:
        m = float(radii.max()) + S_REP + 1.0
        x, y = _place(rng, n, radii, m, nx - 1 - m, max(y_lo * ny, m), ny - 1 - m, S_REP + 1.0)
    P = np.zeros(len(x), lbm.PARTICLE_DTYPE)
    P["x"], P["y"], P["r"] = x, y, radii[: len(x)]
    if shape == "ellipse":
        P["b"] = 0.5 * P["r"]
        P["theta"] = rng.uniform(0.0, math.pi, len(x))
    P["rho"] = 1.5 if setup != "lattice" else 1.1
    P["T"] = rng.uniform(0.8, 1.0, len(x))
    return P


def _params(nu, pr, g, **kw):
    p = dict(nu=nu, alpha=nu / pr, g=g, beta=1.0, T0=0.0, rho_f=1.0, T_init=0.0, s_e=0.0, s_eps=0.0, s_q=0.0, q_e=0.0,
             q_nu=0.0, eps_w=1e-3, s_rep=S_REP, body_fx=0.0, body_fy=0.0, fixed_particles=0)
    p.update(kw)
    return p


def _inputs(case, seed):
    """Inputs of the simulations of a case: a list of (domain, particles, params)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "sim":
        nx, ny, setup = case["nx"], case["ny"], case["setup"]
        P = _particles(rng, nx, ny, case["n"], case["shape"], case["r_lo"], case["r_hi"], case["y_lo"], setup)
        dom = dict(nx=nx, ny=ny, periodic_x=0, periodic_y=0, T_wall=(0.0, 0.0, 0.0, 0.0))
        prm = _params(case["nu"], case["pr"], case["u_ff"] ** 2 / ny * rng.uniform(0.9, 1.0))
        if setup == "bed":
            dom["periodic_x"] = 1
            prm.update(body_fx=1e-6 * rng.uniform(0.5, 1.0), fixed_particles=1)
        if setup == "heated":
            dom["T_wall"] = (1.0, 0.0, 0.5, 0.5)
            prm.update(T_init=0.5, T0=0.5)
        return [(dom, P, prm)]
    out = []
    size = np.random.Generator(np.random.PCG64([case["count"], case["lo"], case["hi"]]))  # the study's, not the seed's
    for _ in range(case["count"]):
        nx, ny = (int(v) for v in size.integers(case["lo"], case["hi"] + 1, 2))
        if case["kind"] == "serve":
            ny = nx
        r = 0.5 * (case["r_lo"] + case["r_hi"])
        room = (nx - 2 * r - 8) * (0.45 * ny - 2 * r - 8)
        n = int(max(1, min(400, size.uniform(0.2, 1.0) * case["fill"] * room / (math.pi * r * r))))
        P = _particles(rng, nx, ny, n, "disk", case["r_lo"], case["r_hi"], 0.5, "settle")
        prm = _params(0.02, 0.71, float(np.exp(rng.uniform(np.log(0.01), np.log(0.04)))) ** 2 / ny)
        out.append((dict(nx=nx, ny=ny, periodic_x=0, periodic_y=0, T_wall=(0.0, 0.0, 0.0, 0.0)), P, prm))
    return out


def _force_inputs(case, seed):
    """A near-rest state around particles that move: FP32 planes, owner map, particles, all on the GPU."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nx, ny = case["nx"], case["ny"]
    P = _particles(rng, nx, ny, case["n"], case["shape"], case["r_lo"], case["r_hi"], 0.05, "settle")
    P["ux"], P["uy"] = rng.normal(0.0, 5e-3, len(P)), rng.normal(0.0, 5e-3, len(P))
    P["omega"] = rng.normal(0.0, 1e-3, len(P))
    pitch = (nx + 31) // 32 * 32
    ps = (pitch * ny + 63) // 64 * 64
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    A = torch.empty((14, ps), dtype=torch.float32, device="cuda").normal_(0.0, 1e-3, generator=gen)
    A[9:].mul_(0.1).add_(torch.tensor([0.3, 0.05, 0.05, 0.05, 0.05], device="cuda")[:, None])
    own = _owner(nx, ny, _columns(P))
    return P, pitch, ps, A, own


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.kind = case["kind"]
    if s.kind == "forces":
        P, s.pitch, s.ps, s.A, own = _force_inputs(case, seed)
        s.nx, s.ny, s.n = case["nx"], case["ny"], len(P)
        s.own = own.to(torch.int32).contiguous()
        s.P = torch.from_numpy(P.view(np.float64).reshape(-1, 10).copy()).cuda()
        s.r_max = float(P["r"].max())
        s.F = torch.zeros((s.n, 3), dtype=torch.float64, device="cuda")
        return s
    if s.kind == "serve":
        s.storage, s.tick = STORAGE[case["storage"]], case["tick"]
        s.requests = [(d, p, q, case["steps"] - 7 * k % 16) for k, (d, p, q) in enumerate(_inputs(case, seed))]
        s.server = lbm.Server(sum(160 * d["nx"] * d["ny"] + 4000 * (len(p) + 64) + (16 << 20)
                                  for d, p, _, _ in s.requests), max_active=max(2, len(s.requests)))
        return s
    s.steps = case["steps"]
    s.sims = [lbm.Simulation(d, p, q, storage=STORAGE[case["storage"]]) for d, p, q in _inputs(case, seed)]
    if s.kind == "sim":
        s.sims[0].step(case["spin"])
    s.parts = [torch.zeros((m.np, 10), dtype=torch.float64, pin_memory=True) for m in s.sims]
    s.views = [t.numpy().reshape(-1).view(lbm.PARTICLE_DTYPE) for t in s.parts]
    if s.kind == "batch":
        s.batch = lbm.Batch(s.sims)
        s.batch.autotune(2)
        nodes = [m.nx * m.ny for m in s.sims]
        s.at = np.concatenate([[0], np.cumsum(nodes)])
        s.fields = [torch.empty(int(s.at[-1]), dtype=torch.float32, device="cuda") for _ in range(4)]
        s.all_parts = torch.zeros((sum(m.np for m in s.sims), 10), dtype=torch.float64, pin_memory=True)
        ends = np.cumsum([0] + [m.np for m in s.sims])
        s.views = [s.all_parts[a:b].numpy().reshape(-1).view(lbm.PARTICLE_DTYPE) for a, b in zip(ends, ends[1:])]
    return s


def run(s):
    if s.kind == "sim":
        sim = s.sims[0]
        sim.step(s.steps)
        f = sim.fields_device()
        if sim.np:
            lbm.lbm_get_particles_async(sim.h, s.views[0])
        return {"drho": f[0], "ux": f[1], "uy": f[2], "T": f[3], "particles": s.parts[0]}
    if s.kind == "batch":
        s.batch.step(s.steps)
        s.batch.sync()
        for m, a, v in zip(s.sims, s.at, s.views):
            lbm.lbm_get_fields(m.h, *[f.data_ptr() + 4 * int(a) for f in s.fields], 1)
            lbm.lbm_get_particles_async(m.h, v)
        return {"fields": s.fields, "particles": s.all_parts}
    if s.kind == "forces":
        lbm.lbm_link_forces_noalloc(s.A.data_ptr(), s.ps, s.pitch, s.own.data_ptr(), s.nx, s.ny, s.P.data_ptr(), s.n,
                                    s.r_max, s.F.data_ptr(), torch.cuda.current_stream().cuda_stream)
        return {"planes": s.A, "forces": s.F}
    ids = [s.server.submit(d, p, q, steps, storage=s.storage) for d, p, q, steps in s.requests]
    while True:
        st = s.server.tick(s.tick)
        if st["active"] == 0 and st["queued"] == 0:
            break
    out = []
    for rid in ids:
        f, p = s.server.result(rid)
        out.append({"drho": f[0], "ux": f[1], "uy": f[2], "T": f[3], "particles": p.view(np.float64).reshape(-1, 10)})
    return out


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Populations read and written once a step (solid nodes left out), fields and particles written once; about
    260 operations a node and step (two MRT collisions) and 90 a link."""
    if case["kind"] == "forces":
        links = case["n"] * 9.85 * (case["r_lo"] + case["r_hi"])
        zone = (case["r_lo"] + case["r_hi"] + 3) ** 2
        return {"bytes": case["n"] * (80 + 24 + 4 * zone) + links * 4 * (5 + 1.6) + links * 5.6, "flops": 90 * links}
    per = 28 if case["storage"] != "fp32" else 56
    total = {"bytes": 0.0, "flops": 0.0}
    for k, (d, p, _) in enumerate(_sizes(case)):
        steps = case["steps"] - (7 * k % 16 if case["kind"] == "serve" else 0)
        nodes = d - p[1]
        total["bytes"] += steps * (2 * per * nodes + 160 * p[0]) + (per + 16) * nodes + 16 * p[1] + 80 * p[0]
        total["flops"] += steps * (260 * nodes + 90 * p[2]) + 30 * nodes
    return total


def _sizes(case):
    """(nodes, (particles, solid nodes, links), unused) of each simulation of a case."""
    def of(n, r, shape):
        f = 0.5 if shape == "ellipse" else 1.0
        return n, n * math.pi * r * r * f, n * 19.7 * r * (0.5 + 0.5 * f)
    if case["kind"] == "sim":
        return [(case["nx"] * case["ny"], of(case["n"], 0.5 * (case["r_lo"] + case["r_hi"]), case["shape"]), None)]
    return [(d["nx"] * d["ny"], of(len(p), float(p["r"].mean()), "disk"), None) for d, p, _ in _inputs(case, 0)]


# ---------------------------------------------------------------------------
# The method in FP64
# ---------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
W5 = (0.6,) + (0.1,) * 4


def _columns(P):
    return {k: torch.from_numpy(np.ascontiguousarray(P[k])).cuda() for k in lbm.PARTICLE_DTYPE.names}


def _is_ell(c):
    return (c["b"] > 0) & (c["b"] != c["r"])


def _frame(c):
    """Semi-axes (a, b) and body axes of each particle, a disk as an ellipse with equal axes."""
    ell = _is_ell(c)
    return c["r"], torch.where(ell, c["b"], c["r"]), torch.cos(c["theta"]), torch.sin(c["theta"]), ell


def _owner(nx, ny, c):
    """Owner map [ny, nx] (int64, -1 fluid): the highest index of the particles that hold a node."""
    own = torch.full((ny * nx,), -1, dtype=torch.int64, device="cuda")
    n = c["x"].numel()
    if n == 0:
        return own.view(ny, nx)
    a, b, cs, sn, ell = _frame(c)
    N = int(torch.ceil(2 * c["r"].max()).item()) + 3
    X0, Y0 = torch.floor(c["x"] - c["r"]).long() - 1, torch.floor(c["y"] - c["r"]).long() - 1
    i = X0[:, None, None] + torch.arange(N, device="cuda")[None, None, :]
    j = Y0[:, None, None] + torch.arange(N, device="cuda")[None, :, None]
    dx, dy = (i.double() - c["x"][:, None, None]), (j.double() - c["y"][:, None, None])
    u, v = dx * cs[:, None, None] + dy * sn[:, None, None], dy * cs[:, None, None] - dx * sn[:, None, None]
    a2, b2 = (a * a)[:, None, None], (b * b)[:, None, None]
    ins = torch.where(ell[:, None, None], (u * u) * b2 + (v * v) * a2 <= a2 * b2, dx * dx + dy * dy <= a2)
    ins &= (i >= 0) & (i < nx) & (j >= 0) & (j < ny)
    who = torch.arange(n, device="cuda")[:, None, None].expand(ins.shape)[ins]
    own.scatter_reduce_(0, (j * nx + i)[ins], who, "amax")
    return own.view(ny, nx)


def _links(A, own, nx, ny, c):
    """Bounce-back values into A [14][ny, nx] at the solid end of every link, and force and torque [n, 3]."""
    n = c["x"].numel()
    F = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    a, b, cs, sn, _ = _frame(c)
    fluid = own < 0
    flat, A2 = fluid.view(-1), A.view(14, -1)

    def inner(i, j):
        ok = (i >= 0) & (i < nx) & (j >= 0) & (j < ny)
        return ok & flat[(j.clamp(0, ny - 1) * nx + i.clamp(0, nx - 1))]

    for k in range(1, 9):
        kx, ky, kb = EX[k], EY[k], OPP[k]
        js, je, is_, ie = max(0, -ky), ny - max(0, ky), max(0, -kx), nx - max(0, kx)
        hit = fluid[js:je, is_:ie] & ~fluid[js + ky:je + ky, is_ + kx:ie + kx]
        at = hit.nonzero()
        if at.numel() == 0:
            continue
        j, i = at[:, 0] + js, at[:, 1] + is_
        n0, ns = j * nx + i, (j + ky) * nx + (i + kx)
        p = own.view(-1)[ns]
        dx, dy = i.double() - c["x"][p], j.double() - c["y"][p]
        ap, bp, cp, sp = a[p], b[p], cs[p], sn[p]
        u, v = dx * cp + dy * sp, dy * cp - dx * sp
        eu, ev = kx * cp + ky * sp, ky * cp - kx * sp
        p2 = (eu / ap) ** 2 + (ev / bp) ** 2
        p1 = u * eu / ap ** 2 + v * ev / bp ** 2
        p0 = (u / ap) ** 2 + (v / bp) ** 2 - 1
        q = (p0 / (-p1 + torch.sqrt((p1 * p1 - p2 * p0).clamp(min=0)))).clamp(max=1)
        h1, h2 = inner(i - kx, j - ky), inner(i - 2 * kx, j - 2 * ky)
        n1, n2 = torch.where(h1, n0 - ky * nx - kx, n0), torch.where(h2, n0 - 2 * (ky * nx + kx), n0)
        fk0, fk1, fk2, fb0, fb1 = A2[k][n0], A2[k][n1], A2[k][n2], A2[kb][n0], A2[kb][n1]
        rx, ry = dx + q * kx, dy + q * ky
        uwx, uwy = c["ux"][p] - c["omega"][p] * ry, c["uy"][p] + c["omega"][p] * rx
        wall = -6 * W9[k] * (kx * uwx + ky * uwy)
        near = torch.where(h1 & h2, q * (2 * q + 1) * fk0 + (1 - 4 * q * q) * fk1 - q * (1 - 2 * q) * fk2 + wall,
                           torch.where(h1, 2 * q * fk0 + (1 - 2 * q) * fk1 + wall, fk0 + wall))
        t = 2 * q - 1
        far = torch.where(h1, fk0 / (q * (2 * q + 1)) + t / q * fb0 - t / (2 * q + 1) * fb1 + wall / (q * (2 * q + 1)),
                          (fk0 + t * fb0 + wall) / (2 * q))
        fnew = torch.where(q <= 0.5, near, far)
        if k <= 4:
            wT = 0.2 * c["T"][p]
            gk0, gk1, gb0 = A2[9 + k][n0], A2[9 + k][n1], A2[9 + kb][n0]
            A2[9 + kb][ns] = torch.where(h1, -gk0 + t / (2 * q + 1) * (gk1 + gb0) + 2 / (2 * q + 1) * wT, -gk0 + wT)
        A2[kb][ns] = fnew
        fk, fb = fk0 + W9[k], fnew + W9[k]
        bx, by = fk * (kx - uwx) - fb * (-kx - uwx), fk * (ky - uwy) - fb * (-ky - uwy)
        F.index_add_(0, p, torch.stack([bx, by, rx * by - ry * bx], 1))
    return F


def _update(c, F, prm, nx, ny):
    """Newton-Euler step with buoyant weight and spring repulsion from walls and other particles."""
    a, b, cs, sn, ell = _frame(c)
    area = math.pi * a * b
    C, M = area * (c["rho"] - prm["rho_f"]) * prm["g"], c["rho"] * area
    I = torch.where(ell, 0.25 * M * (a * a + b * b), 0.5 * M * a * a)

    def reach(who, ux, uy):
        u, v = ux * cs[who] + uy * sn[who], uy * cs[who] - ux * sn[who]
        return torch.sqrt((a[who] * u) ** 2 + (b[who] * v) ** 2)

    def push(gap, scale):
        t = (gap - S_REP) / S_REP
        return torch.where(gap > S_REP, torch.zeros_like(gap), scale / prm["eps_w"] * t * t)

    every = torch.arange(c["x"].numel(), device="cuda")
    one, none = torch.ones_like(a), torch.zeros_like(a)
    hx, hy = reach(every, one, none), reach(every, none, one)
    Fx, Fy = F[:, 0].clone(), F[:, 1] - C
    if not prm["periodic_x"]:
        Fx += push(c["x"] + 0.5 - hx, C) - push(nx - 0.5 - c["x"] - hx, C)
    Fy += push(c["y"] + 0.5 - hy, C) - push(ny - 0.5 - c["y"] - hy, C)
    d2 = (c["x"][:, None] - c["x"]) ** 2 + (c["y"][:, None] - c["y"]) ** 2
    pair = (d2 < (a[:, None] + a + S_REP) ** 2).nonzero()
    pair = pair[pair[:, 0] != pair[:, 1]]
    if pair.numel():
        p, q = pair[:, 0], pair[:, 1]
        dist = torch.sqrt(d2[p, q])
        ux, uy = (c["x"][p] - c["x"][q]) / dist, (c["y"][p] - c["y"][q]) / dist
        mag = push(dist - reach(p, ux, uy) - reach(q, ux, uy), 0.5 * (C[p] + C[q]))
        Fx.index_add_(0, p, mag * ux)
        Fy.index_add_(0, p, mag * uy)
    if prm["fixed_particles"]:
        return c
    ux, uy, om = c["ux"] + Fx / M, c["uy"] + Fy / M, c["omega"] + F[:, 2] / I
    return dict(c, x=c["x"] + 0.5 * (c["ux"] + ux), y=c["y"] + 0.5 * (c["uy"] + uy),
                theta=c["theta"] + 0.5 * (c["omega"] + om), ux=ux, uy=uy, omega=om)


def _pull(A, nx, ny, dom):
    """Streamed populations: half-way bounce-back (flow) and anti-bounce-back (temperature) at walls."""
    S = torch.empty_like(A)
    for p in range(14):
        d = p if p < 9 else p - 9
        kx, ky = EX[d], EY[d]
        S[p] = torch.roll(A[p], (ky, kx), (0, 1))
        back = A[OPP[d] if p < 9 else 9 + OPP[d]]
        side = {1: 0, 3: 1, 2: 2, 4: 3}.get(d, 0)

        def at_wall(rows, cols):
            S[p][rows, cols] = back[rows, cols] if p < 9 else -back[rows, cols] + 2 * W5[d] * dom["T_wall"][side]

        every = slice(None)
        if kx and not dom["periodic_x"]:
            at_wall(every, 0 if kx > 0 else nx - 1)
        if ky and not dom["periodic_y"]:
            at_wall(0 if ky > 0 else ny - 1, every)
    return S


def _refill(S, own, new, nx, ny, c):
    """Newborn nodes: flow extrapolated along the direction nearest the normal, momentum set to the wall's."""
    at = ((own >= 0) & (new < 0)).nonzero()
    if at.numel() == 0:
        return
    j, i = at[:, 0], at[:, 1]
    p = own[j, i]
    a, b, cs, sn, _ = _frame(c)
    dx, dy = i.double() - c["x"][p], j.double() - c["y"][p]
    u, v = (dx * cs[p] + dy * sn[p]) / a[p] ** 2, (dy * cs[p] - dx * sn[p]) / b[p] ** 2
    mx, my = u * cs[p] - v * sn[p], u * sn[p] + v * cs[p]
    ex, ey = torch.tensor(EX, device="cuda"), torch.tensor(EY, device="cuda")
    k = torch.argmax(ex[1:].double() * mx[:, None] + ey[1:].double() * my[:, None], 1) + 1
    uwx, uwy = c["ux"][p] - c["omega"][p] * dy, c["uy"][p] + c["omega"][p] * dx
    calm = ((own < 0) & (new < 0)).view(-1)
    go, f = torch.ones_like(p, dtype=torch.bool), []
    nv = torch.zeros_like(p)
    for m in (1, 2, 3):
        ii, jj = i + m * ex[k], j + m * ey[k]
        go = go & (ii >= 0) & (ii < nx) & (jj >= 0) & (jj < ny)
        node = jj.clamp(0, ny - 1) * nx + ii.clamp(0, nx - 1)
        go = go & calm[node]
        nv += go
        f.append(S.view(14, -1)[:9, node])
    uu = uwx ** 2 + uwy ** 2
    eu = ex[:, None] * uwx + ey[:, None] * uwy
    eq = torch.tensor(W9, dtype=torch.float64, device="cuda")[:, None] * (3 * eu + 4.5 * eu ** 2 - 1.5 * uu)
    fh = torch.where(nv == 3, 3 * f[0] - 3 * f[1] + f[2], torch.where(nv == 2, 2 * f[0] - f[1],
                                                                        torch.where(nv == 1, f[0], eq)))
    rho = 1 + fh.sum(0)
    gx, gy = (rho * uwx - (ex[:, None] * fh).sum(0)) / 6, (rho * uwy - (ey[:, None] * fh).sum(0)) / 6
    S[:9, j, i] = fh + ex[:, None] * gx + ey[:, None] * gy
    w5 = torch.tensor(W5, dtype=torch.float64, device="cuda")[:, None]
    S[9:, j, i] = w5 * c["T"][p] * (1 + 5 * (ex[:5, None] * uwx + ey[:5, None] * uwy))


M9 = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
               [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
               [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], float)
M5 = np.array([[1] * 5, [0, 1, 0, -1, 0], [0, 0, 1, 0, -1], [-4, 1, 1, 1, 1], [0, 1, -1, 1, -1]], float)


def _apply(M, S):
    """M S over the first axis, row by row (S is much larger than M)."""
    out = torch.zeros_like(S)
    for r in range(M.shape[0]):
        for k in range(M.shape[1]):
            if M[r, k]:
                out[r].add_(S[k], alpha=float(M[r, k]))
    return out


def _collide(S, prm):
    """Both MRT collisions; the flow is held as f - w."""
    s_nu = 1 / (3 * prm["nu"] + 0.5)
    rate = [0, 1, 1, 0, 8 * (2 - s_nu) / (8 - s_nu), 0, 8 * (2 - s_nu) / (8 - s_nu), s_nu, s_nu]
    m, T = _apply(M9, S[:9]), S[9:].sum(0)
    rho = 1 + m[0]
    Fx = torch.full_like(rho, prm["body_fx"])
    Fy = rho * prm["g"] * prm["beta"] * (T - prm["T0"]) + prm["body_fy"]
    ux, uy = (m[3] + 0.5 * Fx) / rho, (m[5] + 0.5 * Fy) / rho
    uu, uF = ux * ux + uy * uy, ux * Fx + uy * Fy
    eq = [m[0], -2 * m[0] + 3 * rho * uu, m[0] - 3 * rho * uu, rho * ux, -rho * ux, rho * uy, -rho * uy,
          rho * (ux * ux - uy * uy), rho * ux * uy]
    fm = [0, 6 * uF, -6 * uF, Fx, -Fx, Fy, -Fy, 2 * (ux * Fx - uy * Fy), ux * Fy + uy * Fx]
    for i in range(9):
        m[i] = m[i] - rate[i] * (m[i] - eq[i]) + (1 - 0.5 * rate[i]) * fm[i]
    out = torch.empty_like(S)
    out[:9] = _apply(np.linalg.inv(M9), m)
    k = _apply(M5, S[9:])
    qk = 1 / (prm["alpha"] / 0.2 + 0.5)
    for i, (q, e) in enumerate(((0, T), (qk, T * ux), (qk, T * uy), (1, -2 * T), (1, 0 * T))):
        k[i] = k[i] - q * (k[i] - e)
    out[9:] = _apply(np.linalg.inv(M5), k)
    return out


def _exact_sim(dom, P, prm, steps):
    """Fields and particles after `steps` steps from rest."""
    nx, ny, c = dom["nx"], dom["ny"], _columns(P)
    prm = dict(prm, periodic_x=dom["periodic_x"])
    own = _owner(nx, ny, c)
    A = torch.zeros((14, ny, nx), dtype=torch.float64, device="cuda")
    for k in range(5):
        A[9 + k] = W5[k] * prm["T_init"]
    A = _collide(A, prm)
    A[:, own >= 0] = 0
    for _ in range(steps):
        new = own
        if len(P):
            F = _links(A, own, nx, ny, c)
            c = _update(c, F, prm, nx, ny)
            new = _owner(nx, ny, c)
        S = _pull(A, nx, ny, dom)
        if len(P):
            _refill(S, own, new, nx, ny, c)
        A = _collide(S, prm)
        A[:, new >= 0] = 0
        own = new
    drho, T = A[:9].sum(0), A[9:].sum(0)
    rho = 1 + drho
    jx, jy = (sum(e[k] * A[k] for k in range(1, 9) if e[k]) for e in (EX, EY))
    Fy = rho * prm["g"] * prm["beta"] * (T - prm["T0"]) + prm["body_fy"]
    out = [drho, (jx - 0.5 * prm["body_fx"]) / rho, (jy - 0.5 * Fy) / rho, T]
    for f in out:
        f[own >= 0] = math.nan
    return out, torch.stack([c[k] for k in lbm.PARTICLE_DTYPE.names], 1)


def exact(case, seed):
    if case["kind"] == "forces":
        P, pitch, ps, A, own = _force_inputs(case, seed)
        nx, ny, c = case["nx"], case["ny"], _columns(P)
        B = A[:, : pitch * ny].reshape(14, ny, pitch)[:, :, :nx].double().contiguous()
        F = _links(B, own, nx, ny, c)
        planes = A.double()
        planes[:, : pitch * ny].view(14, ny, pitch)[:, :, :nx] = B
        return {"planes": planes, "forces": F}
    res = []
    for k, (d, p, q) in enumerate(_inputs(case, seed)):
        steps = case["steps"] - (7 * k % 16 if case["kind"] == "serve" else 0)
        f, parts = _exact_sim(d, p, q, steps + (case["spin"] if case["kind"] == "sim" else 0))
        res.append({"drho": f[0], "ux": f[1], "uy": f[2], "T": f[3], "particles": parts})
    if case["kind"] == "sim":
        return res[0]
    if case["kind"] == "serve":
        return res
    return {"fields": [torch.cat([r[k].reshape(-1) for r in res]) for k in ("drho", "ux", "uy", "T")],
            "particles": torch.cat([r["particles"] for r in res])}
