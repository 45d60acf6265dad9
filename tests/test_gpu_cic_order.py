"""The CIC kernels' processing order: in nested systems from 2^16 particles they
run in spatial order, share atomics within runs of one cell and take each point
once per level.  Densities, gradients and trajectories must not depend on it."""
import numpy as np
import pytest

from paper_1210_1736_gb300 import pm, workloads as W
from tests._harness import cast

pytestmark = pytest.mark.gpu


def _case(precision, n, crowd):
    w = W.merger(n_gal=n - 3_000, n_sat=3_000, grids=((32,), (32,), (32, 32, 8), (16,)), seed_id=21,
                 precision=precision, q_m=0.8, r_apo=3.0)
    if crowd:   # runs longer than a warp: a tenth of the points in a few cells
        k = n // 10
        w["pos"][:, :k] = w["pos"][:, :1] + 1e-3 * np.sign(w["pos"][:, :k])
    return w


def _cotangent(w):
    return cast(w, np.random.default_rng(5).normal(size=w["pos"].shape))


def _all(w, perm, u):
    """Densities, accelerations and vector-Jacobian product for the cotangent
    u with the particles stored in the order perm, given back in w's."""
    import torch
    m = cast(w, w["m"])
    ctx = pm.Context(w, W.mass_bound(m))
    p = pm.Particles(cast(w, w["pos"])[:, perm], cast(w, w["vel"])[:, perm], m[perm], w["gal"][perm],
                     precision=w["precision"])
    ctx.cic_deposit(p)
    rho = {k: ctx.density(*k) for k in ctx.shapes}
    ctx.solve()
    acc = torch.stack(ctx.cic_force(p))
    gx, gm = torch.zeros_like(acc), torch.zeros_like(p.m)
    ctx.cic_vjp(p, torch.tensor(u[:, perm], device="cuda").contiguous(), gx, gm)
    back = np.argsort(perm)
    out = [t.cpu().numpy()[..., back] for t in (acc, gx, gm)]
    ctx.close()
    return rho, out


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,crowd", [(1 << 16, False), ((1 << 16) + 1, True), (70_003, False)])
def test_order_changes_nothing(precision, n, crowd):
    w = _case(precision, n, crowd)
    u = _cotangent(w)
    a_rho, a = _all(w, np.arange(n), u)
    b_rho, b = _all(w, np.random.default_rng(3).permutation(n), u)
    for k in a_rho:
        assert np.array_equal(a_rho[k], b_rho[k]), k
    for s, t in zip(a, b):
        assert np.array_equal(s, t)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_ordered_equals_unordered(precision):
    """The same system just below the limit, and above it with massless
    particles without cotangent added: the sums are the same integers, also of
    the adjoint densities where both numbers give one fixed-point scale."""
    n = (1 << 16) - 1
    w = _case(precision, n, True)
    big = dict(w)
    for k in ("pos", "vel"):
        big[k] = np.concatenate([w[k], w[k][:, :500]], axis=1)
    big["m"] = np.concatenate([w["m"], np.zeros(500)])
    big["gal"] = np.concatenate([w["gal"], w["gal"][:500]])
    u = _cotangent(w)
    ub = np.concatenate([u, np.zeros_like(u[:, :500])], axis=1)
    # the scale is 2^(61 - ceil(log2(1.01 n max|u| max(1/l_xy + 1/(2 l_z)))))
    ls = [g for q in w["galaxies"] for g in map(pm.geometry, (q["coarse"], q["medium"], q["fine"]))]
    bound = 1.01 * float(np.abs(u).astype(np.float32).max()) * max(1 / g.l_xy + 1 / (2 * g.l_z) for g in ls)
    assert np.ceil(np.log2(n * bound)) == np.ceil(np.log2((n + 500) * bound))
    a_rho, a = _all(w, np.arange(n), u)
    b_rho, b = _all(big, np.arange(n + 500), ub)
    for k in a_rho:
        assert np.array_equal(a_rho[k], b_rho[k]), k
    for s, t in zip(a, b):   # accelerations, position and mass gradients
        assert s.any() and np.array_equal(s, t[..., :n])


@pytest.mark.parametrize("precision,n", [("fp32", 1 << 16), ("fp32", (1 << 18) - 1), ("fp32", 1 << 18), ("fp64", 1 << 16)])
def test_kick_drift_in_either_order(precision, n):
    """Positions and velocities after a kick-drift, which runs in the stored
    order or in the computed one, do not depend on how particles are stored."""
    w = _case(precision, n, False)
    m, out = cast(w, w["m"]), []
    for perm in (np.arange(n), np.random.default_rng(3).permutation(n)):
        ctx = pm.Context(w, W.mass_bound(m))
        p = pm.Particles(cast(w, w["pos"])[:, perm], cast(w, w["vel"])[:, perm], m[perm], w["gal"][perm],
                         precision=precision)
        ctx.cic_deposit(p)
        ctx.solve()
        ctx.cic_kick_drift(p, 0.01, 0.02)
        pos, vel, _ = p.host()
        back = np.argsort(perm)
        out.append((pos[:, back], vel[:, back]))
        ctx.close()
    assert not np.array_equal(out[0][0], cast(w, w["pos"]))
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_other_particles_of_the_same_number():
    """A call after another set's deposit runs in that set's order: results
    are those of its own particles."""
    import torch
    n = 1 << 16
    w, v = _case("fp32", n, False), _case("fp32", n, True)
    m = cast(w, w["m"])
    ctx = pm.Context(w, W.mass_bound(m))
    ps = [pm.Particles(cast(q, q["pos"]), cast(q, q["vel"]), m, q["gal"]) for q in (w, v)]
    ctx.cic_deposit(ps[0])
    ctx.solve()
    a = torch.stack(ctx.cic_force(ps[1]))    # p1 in p0's order
    ctx2 = pm.Context(w, W.mass_bound(m))
    half = pm.Particles.from_tensors(torch.stack([ps[0].x, ps[0].y, ps[0].z]), torch.stack([ps[0].vx, ps[0].vy, ps[0].vz]),
                                     ps[0].m, ps[0].gal)
    ctx2.cic_deposit(half)
    ctx2.solve()
    k = n - 7                                # another number: as stored
    sub = pm.Particles(cast(v, v["pos"])[:, :k], cast(v, v["vel"])[:, :k], m[:k], v["gal"][:k])
    b = torch.stack(ctx2.cic_force(sub))
    assert torch.equal(a[:, :k], b)


def test_captured_calls_keep_the_stored_order():
    """A captured deposit allocates nothing and its replay gives the ordered
    deposit's densities; a call between capture and replay does not use an
    order that no launch has written."""
    import torch
    n = 1 << 16
    w = _case("fp32", n, False)
    m = cast(w, w["m"])
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = pm.Context(w, W.mass_bound(m))
        p = pm.Particles(cast(w, w["pos"]), cast(w, w["vel"]), m, w["gal"])
        s.synchronize()
        size = ctx.info()["bytes"]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.cic_deposit(p)
        assert ctx.info()["bytes"] == size
        ctx.solve()
        before = torch.stack(ctx.cic_force(p))   # of empty densities
        g.replay()
        captured = {k: ctx.density(*k) for k in ctx.shapes}
        ctx.solve()
        a = torch.stack(ctx.cic_force(p))
        ctx.cic_deposit(p)
        assert ctx.info()["bytes"] == size + 12 * n
        assert all(np.array_equal(captured[k], ctx.density(*k)) for k in ctx.shapes)
        ctx.solve()
        b = torch.stack(ctx.cic_force(p))
        s.synchronize()
    assert not before.any()
    assert a.any() and torch.equal(a, b)
    ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_where_the_order_is_computed(precision):
    """In nested systems from 2^16 particles, and a tenth of the coarse cells
    for a single galaxy in FP32; not on a single grid."""
    import torch

    def grown(w, n):
        ctx = pm.Context(w, W.mass_bound(cast(w, w["m"])))
        p = pm.Particles(cast(w, w["pos"])[:, :n], cast(w, w["vel"])[:, :n], cast(w, w["m"])[:n], w["gal"][:n],
                         precision=precision)
        size = ctx.info()["bytes"]
        ctx.cic_deposit(p)
        ctx.solve()
        a = torch.stack(ctx.cic_force(p))
        assert torch.isfinite(a).all() and a.any()
        size = ctx.info()["bytes"] - size
        ctx.close()
        return size

    n = 1 << 16
    w = _case(precision, n, False)
    assert grown(w, n) == 12 * n and grown(w, n - 1) == 0
    g = W.galaxy_small(precision=precision, n_total=n)
    assert grown(g, n) == 12 * n
    g["galaxies"][0]["coarse"] = (128, 128, 128) + tuple(g["galaxies"][0]["coarse"][3:])
    assert grown(g, n) == (12 * n if precision == "fp64" else 0)
    assert grown(W.big_box(n, 32, precision=precision), n) == 0
