"""Scratch that calls allocate on demand: what a refused allocation leaves
behind, what growth keeps, and the results without memory for it."""
import ctypes as C

import numpy as np
import pytest

from paper_1210_1736_gb300 import pm, workloads as W
from tests._harness import gpu_setup

pytestmark = pytest.mark.gpu


def test_refused_allocation_is_reported_once():
    """A call whose scratch exceeds every memory fails alone; the next call is
    not told of it."""
    w = W.galaxy_small(n_total=4000)
    ctx, p = gpu_setup(w)
    ctx.deposit(p)
    rho = ctx.density(0, 5)
    s = p.struct()
    s.n = 1 << 40   # 4 TiB for the first array: refused before any launch
    assert pm.lib().pm_sort(ctx.h, C.byref(s), None) == pm.PM_E_CUDA
    ctx.deposit(p)
    assert np.array_equal(rho, ctx.density(0, 5))
    ctx.sort(p)
    ctx.close()


def _subset(p, n):
    import torch
    return pm.Particles.from_tensors(torch.stack([p.x, p.y, p.z])[:, :n].contiguous(),
                                     torch.stack([p.vx, p.vy, p.vz])[:, :n].contiguous(), p.m[:n].contiguous(),
                                     p.gal[:n].contiguous())


def test_outgrown_disc_scratch_is_released():
    """The context's bytes follow the largest particle number, not the sum."""
    w = W.galaxy_small(n_total=4000)
    ctx, p = gpu_setup(w)
    base = ctx.info()["bytes"]
    sizes = []
    for n in (1000, 2000, 3000, 3500, 4000, 2500):
        ctx.disc_diagnostics(_subset(p, n))
        sizes.append(ctx.info()["bytes"] - base)
    fixed = sizes[0] - 48 * 1000
    assert 0 < fixed < 1 << 20
    assert sizes == [fixed + 48 * n for n in (1000, 2000, 3000, 3500, 4000, 4000)]
    ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nbins,nring,mmax,nsel", [(1, 1, 1, None), (20, 10, 4, None), (33, 3, 7, 100),
                                                   (64, 16, 64, 5000), (64, 1, 1, 3), (5, 4, 2, 0)])
def test_disc_diagnostics_without_scratch(precision, nbins, nring, mmax, nsel):
    """Without memory for the particles' part the passes read the particles:
    the same bins, the same terms in other sums."""
    import torch
    w = W.galaxy_small(precision=precision, n_total=20_000)
    ctx, p = gpu_setup(w)
    ctx.deposit(p)
    disc = np.asarray(w["comp"]) == W.COMP_DISC
    if nsel is not None:
        disc &= np.cumsum(disc) <= nsel
    sel = torch.tensor(disc, device="cuda")
    out = []
    for limit in (0, -1):
        ctx.selftest_scratch_limit(limit)
        before = ctx.info()["bytes"]
        out.append(ctx.disc_diagnostics(p, sel, nbins=nbins, nring=nring, mmax=mmax)["raw"])
        assert (ctx.info()["bytes"] - before >= 48 * p.n) == (limit < 0)
    counts = slice(7, 6 + 4 * nbins, 4)
    got, ref = out
    assert np.array_equal(got[counts], ref[counts]) and got[0] == ref[0]
    # FP64 sums of at most 20,000 terms in another order (as in test_gpu_diag_paths.py)
    tol = 1e-9 * np.abs(ref) + 1e-12 * np.abs(ref[6 + 4 * nbins:]).max(initial=0.0)
    assert np.all(np.abs(got - ref) <= tol)
    ctx.close()


def test_outgrown_order_is_released_and_refused():
    """The CIC calls' order: 12 bytes for the largest particle number, and the
    same densities and accelerations where it is refused."""
    import torch
    n = (1 << 16) + 3000
    w = W.merger(n_gal=n - 3000, n_sat=3000, grids=((32,), (32,), (32, 32, 8), (16,)), seed_id=21, q_m=0.8, r_apo=3.0)
    ctx, p = gpu_setup(w)
    base = ctx.info()["bytes"]
    for k, cap in ((n - 3000, n - 3000), (n - 2000, n - 2000), (n, n), (n - 1000, n)):
        ctx.cic_deposit(_subset(p, k))
        assert ctx.info()["bytes"] - base == 12 * cap
    res = []
    for limit in (-1, 0):
        ctx, p = gpu_setup(w)
        ctx.selftest_scratch_limit(limit)
        base = ctx.info()["bytes"]
        ctx.cic_deposit(p)
        assert ctx.info()["bytes"] - base == (12 * n if limit < 0 else 0)
        rho = {k: ctx.density(*k) for k in ctx.shapes}
        ctx.solve()
        a = torch.stack(ctx.cic_force(p))
        g, gm = torch.zeros_like(a), torch.zeros_like(p.m)
        ctx.cic_vjp(p, a, g, gm)
        res.append((rho, a, g, gm))
    (ra, *a), (rb, *b) = res
    assert all(np.array_equal(ra[k], rb[k]) for k in ra)
    assert all(torch.equal(s, t) for s, t in zip(a, b))


def test_growth_beside_another_streams_capture():
    """Scratch that grows while the caller captures on another stream neither
    fails nor ends that capture."""
    import torch
    n = (1 << 16) + 2000
    w = W.merger(n_gal=n - 3000, n_sat=3000, grids=((32,), (32,), (32, 32, 8), (16,)), seed_id=21, q_m=0.8, r_apo=3.0)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx, p = gpu_setup(w)
        few = _subset(p, n - 1000)
        ctx.cic_deposit(few)
        s.synchronize()
    t = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    size = ctx.info()["bytes"]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        t.add_(1)
        ctx.cic_deposit(p)   # on s, which is not captured
    assert ctx.info()["bytes"] == size + 12 * 1000
    g.replay()
    g.replay()
    torch.cuda.synchronize()
    assert (t == 2).all()
    rho = {k: ctx.density(*k) for k in ctx.shapes}
    ctx.cic_deposit(p)
    assert all(np.array_equal(rho[k], ctx.density(*k)) for k in ctx.shapes)
