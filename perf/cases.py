"""What users of the particle-mesh library run, as measurable cases.

Every case goes through the library's public entry points (pm.Context,
pm.Particles, adjoint.trajectory and the C call pm_potential_static).  The
particle models are the ones of paper_1210_1736_gb300/workloads.py (a disc, a
bulge and a halo on nested grids, Plummer satellites with their own grids, or
a Plummer sphere on one grid), sampled on the GPU.

Operations ("op"):
  step      leap-frog steps of a running simulation (recentre, deposit, solve,
            kick-drift); with "sort" > 0 the library re-sorts the particles on
            that interval and the particles come back in the caller's order,
            as for a snapshot (their index travels in the caller's bits of the
            flag word)
  field     deposit, solve and the accelerations of a fresh particle set in
            arbitrary order, as before a leap-frog start or for a force probe
  adjoint   forward and backward of a differentiable trajectory
  measure   a snapshot's diagnostics: energies, angular momentum, disc profile
  potential one isolated grid's potential by the allocation-free call
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1210_1736_gb300 import adjoint, pm

RADII = dict(r_core=1.5, r_out=6.0, r_sys=32.0)   # the galaxy's grids
SAT_A, SAT_M = 0.05, 0.1                          # satellite scale length and mass
DT = 0.01


def _case(name, op, prec, n, model="galaxy", nc=32, nm=32, nf=32, nfz=8, sats=0, nsat=0, ns=16, steps=1, sort=0):
    """model "galaxy": n particles on an nc^3 coarse, an nm^3 flattened medium and an nf x nf x nfz fine grid, plus
    `sats` satellites of nsat particles on three ns^3 grids each; model "sphere": n particles on one nc x nm x nf grid
    (fields other than those are not used); op "potential": an nc x nm x nf density of n point masses."""
    return dict(name=name, op=op, prec=prec, model=model, n=n, nc=nc, nm=nm, nf=nf, nfz=nfz, sats=sats, nsat=nsat,
                ns=ns, steps=steps, sort=sort)


def listed():
    return [
        # a test-size galaxy stepped call by call (e.g. coupled to host code each step): launches and latency count
        _case("step_small_fp32", "step", "fp32", 48_000),
        # the convergence run in double precision: one grid, one sphere
        _case("step_sphere_fp64", "step", "fp64", 65_536, model="sphere", nc=32, nm=32, nf=32, steps=10),
        # the ordinary run: 1M particles, ten steps between snapshots, the usual re-sort interval
        _case("step_1m_fp32", "step", "fp32", 1_000_000, nc=128, nm=128, nf=128, nfz=32, steps=10, sort=10),
        # the same run in double precision, the reference for an FP32 production run
        _case("step_1m_fp64", "step", "fp64", 1_000_000, nc=128, nm=128, nf=128, nfz=32, steps=10, sort=10),
        # a galaxy with a sinking satellite
        _case("step_merger_fp32", "step", "fp32", 4_000_000, nc=128, nm=128, nf=256, nfz=32, sats=1, nsat=100_000,
              ns=64, steps=10, sort=10),
        # the largest run of one GPU: 16.5M particles, two satellites, 256^3 grids
        _case("step_large_fp32", "step", "fp32", 16_000_000, nc=256, nm=256, nf=256, nfz=64, sats=2, nsat=250_000,
              ns=128, steps=10, sort=10),
        # initial accelerations of unsorted particles on the largest single grid
        _case("field_box_fp32", "field", "fp32", 1_000_000, model="sphere", nc=256, nm=256, nf=256),
        # a force probe: an odd number of particles, grids of unequal sides, a small satellite
        _case("field_odd_fp32", "field", "fp32", 200_003, nc=64, nm=128, nf=64, nfz=16, sats=1, nsat=5_001, ns=32),
        # gradient check of a small two-galaxy run in double precision
        _case("adjoint_small_fp64", "adjoint", "fp64", 24_000, sats=1, nsat=4_000, ns=32, steps=4),
        # gradients of a production-size trajectory (a segment between checkpoints)
        _case("adjoint_1m_fp32", "adjoint", "fp32", 1_000_000, nc=128, nm=128, nf=128, nfz=32, sats=1, nsat=20_000,
              ns=64, steps=4),
        # diagnostics of a snapshot of the ordinary run
        _case("measure_1m_fp32", "measure", "fp32", 1_000_000, nc=128, nm=128, nf=128, nfz=32),
        # a host application's own density through the allocation-free call
        _case("potential_fp32", "potential", "fp32", 100_000, model="sphere", nc=128, nm=128, nf=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _static_bytes(prec, nx, ny, nz):
    """Upper bound of the allocation-free call's scratch (spectrum, H-hat, its FP64 temporaries), at most 32 MiB."""
    b, P, Q = (4 if prec == "fp32" else 8), nx + 1, ny + 1
    return 8 * b * nx * ny * nz + 2 * b * P * Q * nz + 16 * P * Q * (nz + 1) + 8 * (max(nx, ny, nz) + 1) ** 2 + (1 << 16)


def draw(rng):
    op = rng.choice(["step", "step", "step", "field", "adjoint", "measure", "potential"])
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    if op == "potential":
        sides = [rng.choice([8, 16, 32, 64, 128, 256]) for _ in range(3)]
        while _static_bytes(prec, *sides) > 32 << 20:
            sides[sides.index(max(sides))] //= 2
        return _pure(_case("", op, prec, _log_int(rng, 1000, 200_000), model="sphere", nc=sides[0], nm=sides[1],
                           nf=sides[2]))
    big = prec == "fp32" and op in ("step", "field")
    sides = [32, 64, 128] + ([256] if big else [])
    sort = 10 if op == "step" and rng.random() < 0.7 else 0
    steps = (10 if sort else rng.choice([1, 10])) if op == "step" else rng.randint(1, 4) if op == "adjoint" else 1
    if op in ("step", "field") and rng.random() < 0.25:
        return _pure(_case("", op, prec, _log_int(rng, 4_000, 2_000_000), model="sphere", nc=rng.choice(sides),
                           nm=rng.choice(sides), nf=rng.choice(sides), steps=steps, sort=sort))
    n = _log_int(rng, 10_000, 8_000_000 if big else 900_000)
    nc, nm, nf = (rng.choice(sides) for _ in range(3))
    sats = rng.choice([0, 0, 1, 2]) if big else 0 if prec == "fp64" and max(nc, nm, nf) > 64 else rng.choice([0, 1])
    ns = rng.choice([32, 64] if op == "adjoint" else [16, 32, 64])
    nsat = _log_int(rng, 4_000 if op == "adjoint" else 1_000, max(8_000, n // 10)) if sats else 0
    return _pure(_case("", op, prec, n, nc=nc, nm=nm, nf=nf, nfz=max(8, nf // rng.choice([2, 4, 8] if big else [4, 8])),
                       sats=sats, nsat=nsat, ns=ns, steps=steps, sort=sort))


def _pure(c):
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _interp(x, xp, fp):
    i = torch.searchsorted(xp, x.contiguous()).clamp(1, len(xp) - 1)
    return fp[i - 1] + (fp[i] - fp[i - 1]) * ((x - xp[i - 1]) / (xp[i] - xp[i - 1])).clamp(0, 1)


def _isotropic(g, r):
    c = 2 * torch.rand(r.shape, generator=g, device=r.device, dtype=r.dtype) - 1
    s = torch.sqrt(1 - c * c)
    ph = 2 * math.pi * torch.rand(r.shape, generator=g, device=r.device, dtype=r.dtype)
    return torch.stack([r * s * torch.cos(ph), r * s * torch.sin(ph), r * c])


def _plummer(g, n, M, a, r_trunc):
    f = (r_trunc / a) ** 3 / (1 + (r_trunc / a) ** 2) ** 1.5
    u = (f * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).clamp_min(1e-12)
    r = a / torch.sqrt(u ** (-2.0 / 3.0) - 1)
    sig = torch.sqrt(M / (6 * torch.sqrt(r * r + a * a)))
    vel = sig * torch.randn(3, n, generator=g, device="cuda", dtype=torch.float64)
    return _isotropic(g, r), vel, torch.full((n,), M * f / n, device="cuda", dtype=torch.float64)


def _galaxy(g, n):
    """Exponential sech^2 disc (40 %), Hernquist bulge (10 %), truncated NFW halo (50 %) with velocities of about
    the right size (rotation and dispersions from the spherical enclosed mass)."""
    nd, nb = int(round(0.4 * n)), int(round(0.1 * n))
    nh = n - nd - nb
    kw = dict(device="cuda", dtype=torch.float64)
    Md, Rc, Mb, ab, Mh, rs, rmax = 1.0, 5.0, 0.25, 0.2, 10.0, 3.0, 30.0
    r = torch.logspace(-4, math.log10(rmax), 8001, **kw)

    def disc(x):
        x = x.clamp_max(Rc)
        return (1 - (1 + x) * torch.exp(-x)) / (1 - (1 + Rc) * math.exp(-Rc))

    def halo(x):
        x = x / rs
        return (torch.log1p(x) - x / (1 + x)) / (math.log1p(rmax / rs) - rmax / rs / (1 + rmax / rs))

    bc = 14 * ab / (15 * ab)

    def bulge(x):
        x = x.clamp_max(14 * ab)
        return (x / (x + ab)) ** 2 / bc ** 2

    enc = Md * disc(r) + Mb * bulge(r) + Mh * halo(r)
    vc = lambda q: torch.sqrt(_interp(q, r, enc) / q)   # noqa: E731
    tab = torch.linspace(0, Rc, 20001, **kw)
    R = _interp(torch.rand(nd, generator=g, **kw), disc(tab), tab).clamp_min(1e-3)
    z = 0.1 * torch.atanh(math.tanh(10.0) * (2 * torch.rand(nd, generator=g, **kw) - 1))
    ph = 2 * math.pi * torch.rand(nd, generator=g, **kw)
    c, s = torch.cos(ph), torch.sin(ph)
    w = torch.randn(3, nd, generator=g, **kw)
    v = vc(R)
    vR, vp = 0.15 * v * w[0], v * (0.95 + 0.1 * w[1])
    pos = [torch.stack([R * c, R * s, z])]
    vel = [torch.stack([vR * c - vp * s, vR * s + vp * c, 0.12 * v * w[2]])]
    su = bc * torch.sqrt(torch.rand(nb, generator=g, **kw).clamp_min(1e-9))
    rb = ab * su / (1 - su)
    rh = _interp(torch.rand(nh, generator=g, **kw), halo(r), r).clamp_min(1e-4)
    for q in (rb, rh):
        pos.append(_isotropic(g, q))
        vel.append(vc(q) / math.sqrt(3.0) * torch.randn(3, q.shape[0], generator=g, **kw))
    m = torch.cat([torch.full((k,), M / max(k, 1), **kw) for k, M in ((nd, Md), (nb, Mb), (nh, Mh))])
    return torch.cat(pos, 1), torch.cat(vel, 1), m


def _inputs(case, seed):
    """The workload (grids) and the particles: pos (3, n), vel (3, n), m, gal, disc (the diagnostics' selection), in
    the context's precision and an order of no meaning."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (seed + 1))
    dt = torch.float32 if case["prec"] == "fp32" else torch.float64
    if case["model"] == "sphere":
        # a Plummer sphere that fills the usable box of the smallest side
        sides = (case["nc"], case["nm"], case["nf"])
        R = 3.5
        l_min = 2 * R / (case["nc"] - 4)
        r_box = l_min * (min(sides) / 2 - 3)
        a = r_box / 3.375   # its mass a^3 keeps the dynamical time of M = a = 1
        pos, vel, m = _plummer(g, case["n"], a ** 3, a, 0.99 * r_box)
        gal = torch.zeros(case["n"], dtype=torch.int32, device="cuda")
        gals = [dict(coarse=(*sides, R, 1.0), medium=None, fine=None, r_core=0.0, r_out=0.0, centre=(0.0, 0.0, 0.0),
                     recentre=False)]
        nd = case["n"]
        r_sys = r_box
    else:
        pos, vel, m = _galaxy(g, case["n"])
        nd = int(round(0.4 * case["n"]))
        gal = [torch.zeros(case["n"], dtype=torch.int32, device="cuda")]
        q = {32: 0.8, 64: 0.4}.get(case["nm"], 0.25)   # admissible flattening of the medium grid
        gals = [dict(coarse=(case["nc"],) * 3 + (RADII["r_sys"], 1.0), medium=(case["nm"],) * 3 + (RADII["r_out"], q),
                     fine=(case["nf"], case["nf"], case["nfz"], RADII["r_core"], 1.0), r_core=RADII["r_core"],
                     r_out=RADII["r_out"], centre=(0.0, 0.0, 0.0), recentre=True)]
        allp, allv, allm = [pos], [vel], [m]
        for k in range(case["sats"]):
            ps, vs, ms = _plummer(g, case["nsat"], SAT_M, SAT_A, 10 * SAT_A)
            R, phase, inc = (8.0, 0.0, math.radians(30)) if k == 0 else (6.0, 2.0, math.radians(-45))
            c, s = math.cos(phase), math.sin(phase)
            va = math.sqrt(6.0 * 0.5 / R)
            cen = (R * c, R * s, 0.0)
            add = lambda a, b: a + torch.tensor(b, device="cuda", dtype=torch.float64)[:, None]   # noqa: E731
            allp.append(add(ps, cen))
            allv.append(add(vs, (-s * va * math.cos(inc), c * va * math.cos(inc), va * math.sin(inc))))
            allm.append(ms)
            gal.append(torch.full((case["nsat"],), k + 1, dtype=torch.int32, device="cuda"))
            gals.append(dict(coarse=(case["ns"],) * 3 + (RADII["r_sys"], 1.0),
                             medium=(case["ns"],) * 3 + (10 * SAT_A, 1.0), fine=(case["ns"],) * 3 + (2.5 * SAT_A, 1.0),
                             r_core=2.5 * SAT_A, r_out=10 * SAT_A, centre=cen, recentre=True))
        pos, vel, m, gal = torch.cat(allp, 1), torch.cat(allv, 1), torch.cat(allm), torch.cat(gal)
        r_sys = RADII["r_sys"]
    order = torch.randperm(pos.shape[1], generator=g, device="cuda")
    disc = order < nd
    pos, vel, m, gal = pos[:, order].to(dt), vel[:, order].to(dt), m[order].to(dt), gal[order]
    w = dict(name="case", precision=case["prec"], dt=DT, steps=1,
             system=dict(r_sys=r_sys, sys_centre=(0.0, 0.0, 0.0), G=1.0, h000=1.0), galaxies=gals)
    return w, pos.contiguous(), vel.contiguous(), m.contiguous(), gal.contiguous(), disc


def _cotangents(case, pos, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(7 * seed + 5)
    return torch.randn(2, *pos.shape, generator=g, device="cuda", dtype=torch.float64).to(pos.dtype)


def _density(case, seed):
    """The density a host application hands over: fixed-point masses of point masses, and the grid."""
    w, pos, _, m, _, _ = _inputs(case, seed)
    gm = _Geom(w["galaxies"][0]["coarse"])
    shift = 60
    q = torch.round(torch.ldexp(m.double(), torch.tensor(shift, device="cuda"))).to(torch.int64)
    (i, j, k), ok = _cells(gm, [_off(pos[a], 0.0, case["prec"] == "fp32") for a in range(3)])
    rho = torch.zeros(gm.nz * gm.ny * gm.nx, dtype=torch.int64, device="cuda")
    rho.index_add_(0, ((k * gm.ny + j) * gm.nx + i)[ok], q[ok])
    return gm, rho, shift


def prepare(case, seed):
    st = dict(op=case["op"], steps=case["steps"])
    if case["op"] == "potential":
        gm, rho, shift = _density(case, seed)
        f32 = case["prec"] == "fp32"
        st.update(gm=gm, rho=rho, shift=shift, precision=pm.PM_FP32 if f32 else pm.PM_FP64,
                  phi=torch.empty(gm.nz, gm.ny, gm.nx, device="cuda", dtype=torch.float32 if f32 else torch.float64))
        return st
    w, pos, vel, m, gal, disc = _inputs(case, seed)
    ctx = pm.Context(w, float(m.double().abs().sum()))
    st["ctx"] = ctx
    if case["op"] == "adjoint":
        st.update(x=pos.requires_grad_(True), v=vel.requires_grad_(True), m=m.requires_grad_(True),
                  runner=adjoint.Runner(ctx, gal, DT, case["steps"]), cot=_cotangents(case, pos.detach(), seed))
        return st
    flags = torch.arange(pos.shape[1], dtype=torch.int32, device="cuda") << 1 if case["sort"] else None
    st["p"] = pm.Particles.from_tensors(pos, vel, m, gal, flags)
    st["sort"] = case["sort"]
    if case["op"] == "step" and case["sort"]:
        ctx.set_sort_interval(case["sort"])
    st["disc"] = disc
    return st


def run(st):
    op = st["op"]
    if op == "potential":
        gm, phi = st["gm"], st["phi"]
        rc = pm.lib().pm_potential_static(st["rho"].data_ptr(), phi.data_ptr(), gm.nx, gm.ny, gm.nz, gm.lxy, gm.lz, 1.0,
                                          1.0, st["shift"], st["precision"], torch.cuda.current_stream().cuda_stream)
        if rc != pm.PM_OK:
            raise RuntimeError(pm.lib().pm_last_error().decode())
        return phi
    ctx = st["ctx"]
    if op == "adjoint":
        x, v = adjoint.trajectory(st["x"], st["v"], st["m"], st["runner"])
        g = torch.autograd.grad((x, v), (st["x"], st["v"], st["m"]), (st["cot"][0], st["cot"][1]))
        return dict(x=x.detach(), v=v.detach(), gx=g[0], gv=g[1], gm=g[2])
    p = st["p"]
    if op == "field":
        ctx.deposit(p)
        ctx.solve()
        return torch.stack(ctx.force(p))
    if op == "measure":
        e = ctx.diagnostics(p, DT)
        d = ctx.disc_diagnostics(p, select=st["disc"])
        one = np.atleast_1d
        return dict(K=one(e["K"]), W=one(e["W"]), L=e["L"], n=e["n_live"], heat=one(d["E_heat"]),
                    sigma=np.array([d["sigma_R"], d["sigma_phi"], d["sigma_z"]]), R=d["R_mean"],
                    count=d["count"].astype(np.int64), z=d["z_rms"], vc=d["v_c"], A=d["A"])
    ctx.step(p, DT, st["steps"])
    out = (p.x, p.y, p.z, p.vx, p.vy, p.vz)
    if st["sort"]:
        # back to the caller's order
        ids = (p.flags >> 1).long()
        new = torch.empty(6, p.n, dtype=p.dtype, device="cuda")
        for k in range(6):
            new[k, ids] = out[k]
        return dict(x=new[:3], v=new[3:])
    return dict(x=torch.stack(out[:3]), v=torch.stack(out[3:]))


# ---------------------------------------------------------------------------
# work and tolerances
# ---------------------------------------------------------------------------
def work(case):
    b = 4 if case["prec"] == "fp32" else 8
    if case["op"] == "potential":
        A = case["nc"] * case["nm"] * case["nf"]
        return {"bytes": A * (8 + b), "flops": 3 * 2.5 * 8 * A * math.log2(8 * A)}
    n = case["n"] + case["sats"] * case["nsat"]
    # per grid of one galaxy: cells times real transforms (forward and inverse of each mass set)
    if case["model"] == "sphere":
        grids = [(case["nc"] * case["nm"] * case["nf"], 1)]
    else:
        grids = [(case["nc"] ** 3, 2), (case["nm"] ** 3, 2), (case["nf"] ** 2 * case["nfz"], 1)]
        grids += case["sats"] * [(case["ns"] ** 3, 2), (case["ns"] ** 3, 2), (case["ns"] ** 3, 1)]
    solve = sum(k * 2 * 2.5 * 8 * A * math.log2(8 * A) for A, k in grids)
    hhat = b * sum(A for A, _ in grids)
    # particles in (3 positions, 3 velocities, mass, galaxy, flag) and out, the Green's function per solve
    if case["op"] == "step":
        s = case["steps"]
        return {"bytes": s * (n * (13 * b + 8) + hhat), "flops": s * (solve + 300.0 * n)}
    if case["op"] == "field":
        return {"bytes": n * (7 * b + 8) + hhat, "flops": solve + 300.0 * n}
    if case["op"] == "measure":
        return {"bytes": n * (7 * b + 9) + hhat, "flops": solve + 500.0 * n}
    s = case["steps"]
    # forward: steps + 2 forces; backward: recomputed forces and, per force, its transposed solve
    return {"bytes": (4 * s + 6) * (n * 10 * b + hhat), "flops": (4 * s + 6) * (solve + 600.0 * n)}


def tolerance(case):
    """About four times the largest difference from the same in 64 bits seen over the listed and drawn cases.  FP32
    errors are the FFTs' rounding of the potentials; a step's `max` is a particle whose rounded position falls in
    another cell or region than in 64 bits, a gradient's is set by the second differences of a deep FP32 potential."""
    f32 = case["prec"] == "fp32"
    if case["op"] == "step":
        return {"rel": 5e-5, "max": 4e-2} if f32 else {"rel": 4e-13, "max": 4e-12}
    if case["op"] == "field":
        return {"rel": 4e-5, "max": 4e-4} if f32 else {"rel": 5e-13, "max": 2e-12}
    if case["op"] == "potential":
        return {"rel": 5e-7, "max": 3e-6} if f32 else {"rel": 2e-15, "max": 1e-14}
    if case["op"] == "measure":
        return {"rel": 3e-7} if f32 else {"rel": 2e-13}
    return {"rel": 1.6e-4, "max": 0.24} if f32 else {"rel": 2e-10, "max": 1e-9}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------
class _Geom:
    def __init__(self, spec):
        self.nx, self.ny, self.nz, R, q = spec
        self.lxy = 2.0 * R / (self.nx - 4)
        self.lz = q * self.lxy
        self.l = (self.lxy, self.lxy, self.lz)
        self.n = (self.nx, self.ny, self.nz)
        self._hat = None

    def potential(self, rho):
        """G = 1, H(0,0,0) = 1: the isolated convolution on the doubled grid."""
        s = (2 * self.nz, 2 * self.ny, 2 * self.nx)
        if self._hat is None:
            ax = [torch.minimum(torch.arange(k, device="cuda"), k - torch.arange(k, device="cuda")).double() for k in s]
            h = ((ax[0] * (self.lz / self.lxy))[:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2] ** 2).rsqrt()
            h[0, 0, 0] = 1.0
            self._hat = torch.fft.rfftn(h).real.contiguous()
            del h
        f = torch.fft.irfftn(torch.fft.rfftn(rho.reshape(self.nz, self.ny, self.nx), s=s) * self._hat, s=s)
        return f[:self.nz, :self.ny, :self.nx].contiguous() / self.lxy


def _off(x, c, split):
    """The library's FP32 offset from a centre (its cell assignment is defined by it)."""
    if not split:
        return (x - c).float()
    hi = np.float32(c)
    lo = np.float32(float(c) - float(hi))
    return (x.float() - float(hi)) - float(lo)


def _cells(gm, d):
    idx, ok = [], None
    for k in range(3):
        f = torch.tensor(1.0 / gm.l[k], dtype=torch.float32, device="cuda")
        a = torch.floor((d[k] * f + float(gm.n[k] // 2)) + 0.5).long()
        idx.append(a)
        o = (a >= 2) & (a <= gm.n[k] - 3)
        ok = o if ok is None else ok & o
    return idx, ok


def _r2(d):
    return (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]


class _System:
    """Mass sets, combination rule and both force schemes of a workload, in 64 bits."""

    def __init__(self, w, m):
        self.shift = torch.tensor(62 - math.ceil(math.log2(float(m.abs().sum()))), device="cuda")
        self.split = w["precision"] == "fp32"
        self.r_sys = w["system"]["r_sys"]
        geoms = {}
        mk = lambda s: None if s is None else geoms.setdefault(tuple(s), _Geom(s))   # noqa: E731
        self.gal = [dict(coarse=mk(g["coarse"]), med=mk(g["medium"]), fine=mk(g["fine"]), rc=g["r_core"], ro=g["r_out"],
                         move=g["recentre"]) for g in w["galaxies"]]
        self.cen = [list(g["centre"]) for g in w["galaxies"]]

    def offs(self, x, c):
        x = x.detach()
        return [_off(x[k], c[k], self.split) for k in range(3)]

    def lost(self, x, lost):
        d = self.offs(x, (0.0, 0.0, 0.0))
        lost = lost | ~(_r2(d) < float(np.float32(self.r_sys * self.r_sys)))
        for g in self.gal:
            lost = lost | ~_cells(g["coarse"], d)[1]
        return lost

    def region(self, x, g):
        G = self.gal[g]
        d = self.offs(x, self.cen[g])
        r2 = _r2(d)
        reg = torch.full(r2.shape, 2, dtype=torch.int8, device="cuda")
        if G["med"] is None:
            return reg
        ok2 = _cells(G["med"], d)[1]
        shell = (r2 < float(np.float32(G["ro"] ** 2))) & ok2
        reg[shell] = 1
        if G["fine"] is not None:
            reg[(r2 < float(np.float32(G["rc"] ** 2))) & ok2 & _cells(G["fine"], d)[1]] = 0
        return reg

    def recentre(self, x, m, gal, lost):
        for g, G in enumerate(self.gal):
            if not G["move"]:
                continue
            d = self.offs(x, self.cen[g])
            s = (gal == g) & ~lost & (_r2(d) < float(np.float32(G["rc"] ** 2)))
            # the library's integer centre of mass: weights to 36 bits, offsets to 24 bits of R_core
            M = torch.round(torch.ldexp(m[s], self.shift)).long() >> 26
            sD = 24 - math.ceil(math.log2(G["rc"]))
            D = [torch.round(d[k][s] * 2.0 ** sD).long() for k in range(3)]
            if int(M.sum()) > 0:
                self.cen[g] = [self.cen[g][k] + int((M * D[k]).sum()) / int(M.sum()) * 2.0 ** -sD for k in range(3)]

    def at(self, gm, x, c):
        """NGP cells and the offsets from their centres."""
        idx, _ = _cells(gm, self.offs(x, c))
        return idx, [x[k] - c[k] - (idx[k] - gm.n[k] // 2).double() * gm.l[k] for k in range(3)]

    def corners(self, gm, x, c):
        """The 8 cloud-in-cell cells and their trilinear weights."""
        idx, dl = self.at(gm, x, c)
        lo, t = [], []
        for k in range(3):
            f = dl[k] / gm.l[k]
            neg = f.detach() < 0
            lo.append(idx[k] - neg.long())
            t.append(f + neg.double())
        for dk in (0, 1):
            for dj in (0, 1):
                for di in (0, 1):
                    w = (t[0] if di else 1 - t[0]) * (t[1] if dj else 1 - t[1]) * (t[2] if dk else 1 - t[2])
                    yield ((lo[2] + dk) * gm.ny + lo[1] + dj) * gm.nx + lo[0] + di, w

    def deposit(self, gm, x, c, m, cic):
        rho = torch.zeros(gm.nz * gm.ny * gm.nx, dtype=torch.float64, device="cuda")
        if not cic:
            idx, _ = _cells(gm, self.offs(x, c))
            return rho.index_add(0, (idx[2] * gm.ny + idx[1]) * gm.nx + idx[0], m)
        for at, w in self.corners(gm, x, c):
            rho = rho.index_add(0, at, m * w)
        return rho

    def force(self, gm, phi, x, c, cic):
        """Acceleration (3, n) and potential of one grid at x."""
        if cic:
            g = [(torch.roll(phi, -1, 2 - k) - torch.roll(phi, 1, 2 - k)).reshape(-1) / (2 * gm.l[k]) for k in range(3)]
            a = torch.zeros_like(x)
            for at, w in self.corners(gm, x, c):
                a = a + torch.stack([w * g[k][at] for k in range(3)])
            return a, None
        idx, d = self.at(gm, x, c)
        f = phi.reshape(-1)
        st = (1, gm.nx, gm.nx * gm.ny)
        o = idx[0] + gm.nx * (idx[1] + gm.ny * idx[2])
        at = lambda *s: f[o + sum(s)]   # noqa: E731
        p0 = at()
        grad, a = [], []
        for k in range(3):
            p, q = at(st[k]), at(-st[k])
            grad.append((p - q) / (2 * gm.l[k]))
            a.append(grad[k] + (p + q - 2 * p0) / gm.l[k] ** 2 * d[k])
        for i, j in ((0, 1), (0, 2), (1, 2)):
            mix = (at(st[i], st[j]) - at(-st[i], st[j]) + at(-st[i], -st[j]) - at(st[i], -st[j])) / (4 * gm.l[i] * gm.l[j])
            a[i] = a[i] + mix * d[j]
            a[j] = a[j] + mix * d[i]
        return torch.stack(a), p0 + grad[0] * d[0] + grad[1] * d[1] + grad[2] * d[2]

    def accel(self, x, m, gal, lost, cic=False):
        """Accelerations (0 for lost particles) and potentials, by the combination rule over every galaxy."""
        zero = (0.0, 0.0, 0.0)
        live = torch.nonzero(~lost)[:, 0]
        acc, pot = torch.zeros_like(x), torch.zeros_like(x[0])
        for g, G in enumerate(self.gal):
            reg = self.region(x, g)
            own = live[gal[live] == g]
            C, M, F, cen = G["coarse"], G["med"], G["fine"], self.cen[g]
            sel = lambda pool, *r: pool[sum((reg[pool] == k) for k in r).bool()]   # noqa: E731

            def phi(gm, c, *r):
                s = sel(own, *r)
                return gm.potential(self.deposit(gm, x[:, s], c, m[s], cic))

            # region: the grids whose potentials act there
            p5 = phi(C, zero, 2)
            parts = []
            if M is None:
                parts.append(((2,), C, zero, p5))
            else:
                parts.append(((2,), C, zero, p5 + phi(C, zero, 0, 1)))
                parts.append(((0, 1), C, zero, p5))
                p3 = phi(M, cen, 1)
                parts.append(((1,), M, cen, p3 + phi(M, cen, 0)))
                parts.append(((0,), M, cen, p3))
                if F is not None:
                    parts.append(((0,), F, cen, phi(F, cen, 0)))
            for r, gm, c, f in parts:
                s = sel(live, *r)
                if len(s):
                    a, q = self.force(gm, f, x[:, s], c, cic)
                    acc = acc.index_add(1, s, a)
                    pot = pot if q is None else pot.index_add(0, s, q)
        return acc, pot


def exact(case, seed):
    if case["op"] == "potential":
        gm, rho, shift = _density(case, seed)
        return gm.potential(torch.ldexp(rho.double(), torch.tensor(-shift, device="cuda")))
    w, pos, vel, m, gal, disc = _inputs(case, seed)
    x, v, m = pos.double(), vel.double(), m.double()
    S = _System(w, m)
    lost = torch.zeros(m.shape, dtype=torch.bool, device="cuda")
    if case["op"] == "field":
        return S.accel(x, m, gal, S.lost(x, lost))[0]
    if case["op"] == "step":
        for _ in range(case["steps"]):
            S.recentre(x, m, gal, lost)
            lost = S.lost(x, lost)
            a, _ = S.accel(x, m, gal, lost)
            # the state is held in the run's type between steps
            v = (v + DT * a).to(pos.dtype).double()
            x = (x + DT * torch.where(lost, torch.zeros_like(v), v)).to(pos.dtype).double()
        return dict(x=x, v=v)
    if case["op"] == "adjoint":
        leaf = [t.clone().requires_grad_(True) for t in (x, v, m)]
        x, v, m = leaf

        def kick(dt):
            nonlocal lost
            lost = S.lost(x, lost)
            return torch.where(lost, torch.zeros_like(v), dt * S.accel(x, m, gal, lost, cic=True)[0])

        # the state is held in the run's type between steps (its rounding has the identity's gradient)
        hold = lambda q: q + (q.to(pos.dtype).double() - q).detach()   # noqa: E731
        v = hold(v + kick(-0.5 * DT))
        for _ in range(case["steps"]):
            v = hold(v + kick(DT))
            x = hold(x + DT * torch.where(lost, torch.zeros_like(v), v))
        v = v + kick(0.5 * DT)
        cot = _cotangents(case, pos, seed).double()
        g = torch.autograd.grad((x, v), leaf, (cot[0], cot[1]))
        return dict(x=x.detach(), v=v.detach(), gx=g[0], gv=g[1], gm=g[2])
    # measure
    lost = S.lost(x, lost)
    a, pot = S.accel(x, m, gal, lost)
    h = ~lost
    xl, ml = x[:, h], m[h]
    vl = v[:, h] + 0.5 * DT * a[:, h]
    out = dict(K=0.5 * (ml * (vl * vl).sum(0)).sum()[None], W=-0.5 * (ml * pot[h]).sum()[None],
               L=(ml * torch.cross(xl, vl, dim=0)).sum(1), n=int(h.sum()))
    s = h & disc
    d, u, md = x[:, s], v[:, s], m[s]
    R2 = d[0] * d[0] + d[1] * d[1]
    R = torch.sqrt(R2)
    n, B = int(s.sum()), 20
    edges = torch.sort(R2)[0][[(k * n) // B for k in range(1, B)]]
    b = torch.searchsorted(edges, R2, right=True)
    add = lambda q: torch.zeros(B, dtype=torch.float64, device="cuda").index_add(0, b, q)   # noqa: E731
    vR, vp = (d[0] * u[0] + d[1] * u[1]) / R, (d[0] * u[1] - d[1] * u[0]) / R
    cnt = add(torch.ones_like(R))
    out["count"] = cnt.long()
    out["R"], out["z"], out["vc"] = add(R) / cnt, torch.sqrt(add(d[2] * d[2]) / cnt), add(vp) / cnt
    xp, fp = out["R"], out["vc"]
    vb = _interp(R, xp, fp)
    out["heat"] = (0.5 * md * (vR * vR + (vp - vb) ** 2 + u[2] * u[2])).sum()[None]
    ring = (R >= 3.2 - 0.4) & (R < 3.2 + 0.4)
    wr = md[ring] / md[ring].sum()
    out["sigma"] = torch.stack([torch.sqrt((wr * q[ring] ** 2).sum() - (wr * q[ring]).sum() ** 2) for q in (vR, vp, u[2])])
    k = torch.floor(R / 0.5).long()
    inr = (R > 0) & (R < 5.0) & (k < 10)
    z = torch.complex(d[0][inr] / R[inr], -d[1][inr] / R[inr])
    A = []
    for mo in range(1, 5):
        q = md[inr] * z ** mo
        re, im = (torch.zeros(10, dtype=torch.float64, device="cuda").index_add(0, k[inr], t) for t in (q.real, q.imag))
        A.append(torch.complex(re, im))
    r = torch.arange(10, dtype=torch.float64, device="cuda") * 0.5
    out["A"] = torch.stack(A, 1) / (math.pi * ((r + 0.5) ** 2 - r ** 2))[:, None]
    return out
