"""The FP64 transforms run in block floating point (pm_fx.cuh): exponents,
zeros and values that overflow, where the arithmetic differs from FP64's."""
import numpy as np
import pytest

from paper_1210_1736_gb300 import pm, workloads as W

pytestmark = pytest.mark.gpu


def _potential(w, G=1.0, mb=None, pos=None, m=None):
    ww = dict(w, system=dict(w["system"], G=G))
    m = w["m"] if m is None else m
    ctx = pm.Context(ww, W.mass_bound(m) if mb is None else mb)
    p = pm.Particles(w["pos"] if pos is None else pos, w["vel"], m, w["gal"], precision="fp64")
    ctx.deposit(p)
    ctx.solve()
    out = {key: ctx.potential(*key) for key in ctx.shapes}
    ctx.close()
    return out


def _box(nx, ny, nz, n=2000):
    w = W.big_box(n, 64, precision="fp64")
    g = w["galaxies"][0]
    g["coarse"] = (nx, ny, nz, g["coarse"][3], 1.0)
    w["system"]["r_sys"] = 0.8 * pm.cell_length(g["coarse"][3], nx) * (min(nx, ny, nz) / 2 - 3)
    return w


@pytest.mark.parametrize("shape", [(8, 16, 32), (64, 8, 128), (16, 256, 8), (256, 8, 64), (8, 64, 256)])
@pytest.mark.parametrize("k", [-820, -400, 31, 600, 820])
def test_scale_invariance(shape, k):
    """G 2^k scales every intermediate by 2^k exactly, also where a group's
    exponent leaves the fast path of the conversion."""
    w = _box(*shape)
    a, b = _potential(w)[(0, 5)], _potential(w, G=2.0 ** k)[(0, 5)]
    assert np.abs(a).max() > 0
    assert np.array_equal(np.ldexp(a, k), b)


def test_nested_scale_invariance():
    """Grid 1's difference-field pass too."""
    w = W.galaxy_small(precision="fp64", n_total=4000)
    a, b = _potential(w), _potential(w, G=2.0 ** -300)
    for key in a:
        assert np.array_equal(np.ldexp(a[key], -300), b[key]), key


def test_empty_density_is_zero():
    w = _box(32, 16, 8)
    p = _potential(w, pos=w["pos"] + 1e6)[(0, 5)]   # every particle lost
    assert np.array_equal(p, np.zeros_like(p))


def test_overflow_is_not_finite():
    """A Green's function beyond the FP64 range gives no finite potential."""
    w = _box(16, 16, 16)
    with np.errstate(over="ignore"):
        p = _potential(w, G=1e308, m=w["m"] * 1e6)[(0, 5)]
    assert not np.isfinite(p).any()


@pytest.mark.parametrize("heavy", [True, False])
@pytest.mark.parametrize("shape", [(32, 32, 32), (128, 16, 16), (16, 16, 256)])
def test_mass_range(shape, heavy):
    """Masses of 2^-40 of the mass bound, whose integer densities have few
    bits, alone and beside one heavy cell."""
    import oracle as O
    w = _box(*shape)
    m = w["m"] * 2.0 ** -40
    mb = W.mass_bound(w["m"])
    pos = w["pos"].copy()
    pos[:, 0] = 0.0
    if heavy:
        m[0] = w["m"][0]
    p = _potential(w, m=m, mb=mb, pos=pos)[(0, 5)]
    ww = dict(w, m=m, pos=pos)
    s = O.system_from_workload(ww, mb)
    st = O.state_from_workload(ww)
    rho, flags, sh = O.deposit(st, s)
    ref = O.solve_all(rho, s, sh)[0][5]
    # both sides round the stored passes and numpy's every operation: a few
    # units of 2^-53 of the largest value
    assert np.abs(p - ref).max() <= 16 * 2.0 ** -53 * np.abs(ref).max()


def _static(rho, shape, shift=50, G=1.0, h000=1.0, precision=pm.PM_FP64):
    """pm_potential_static of a host int64 density [z][y][x]."""
    import torch
    nx, ny, nz = shape
    r = torch.tensor(rho, device="cuda")
    phi = torch.empty(nz, ny, nx, device="cuda", dtype=torch.float64 if precision == pm.PM_FP64 else torch.float32)
    st = torch.cuda.current_stream().cuda_stream
    pm._check(pm.lib().pm_potential_static(r.data_ptr(), phi.data_ptr(), nx, ny, nz, 0.5, 0.25, G, h000, shift, precision, st))
    pm._check(pm.lib().pm_potential_static_status(st))
    return phi.cpu().numpy()


@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 32, 32)])   # whole and half spectra
@pytest.mark.parametrize("near", [0, 3, 7, 8, 9, 40])
@pytest.mark.parametrize("sign", [1, -1])
def test_densities_up_to_the_integer_limits(shape, near, sign):
    """Cells within a rounding unit of +-2^63, alone and beside small ones."""
    nx, ny, nz = shape
    rng = np.random.default_rng(4)
    rho = rng.integers(-2 ** 40, 2 ** 40, size=(nz, ny, nx))
    big = rho.copy()
    for cell in ((0, 0, 0), (3, 5, 7), (nz - 1, ny - 1, nx - 1)):
        big[cell] = 2 ** 63 - 1 - near if sign > 0 else -2 ** 63 + near
    # the same to a relative 2^-59: heavy cells of 2^62, twice, as the potential is linear
    heavy = np.where(big == rho, 0, sign * 2 ** 62)
    a, b = _static(big, shape), 2.0 * _static(heavy, shape) + _static(np.where(big == rho, rho, 0), shape)
    # three potentials, each within 16 units of 2^-53 of the largest value (see test_mass_range)
    assert np.abs(a - b).max() <= 48 * 2.0 ** -53 * np.abs(b).max()


# tiles wider than the grid (their warps beyond it hold zeros), whole and half spectra
@pytest.mark.parametrize("shape", [(16, 16, 16), (8, 16, 8), (16, 8, 8), (64, 32, 32), (8, 64, 16)])
@pytest.mark.parametrize("G,shift", [(-880, 50), (-925, 50), (-960, 50), (-975, 50), (900, 1000), (-960, -20)])
def test_small_magnitudes(shape, G, shift):
    """Green's functions and masses towards the least FP64 exponents: the
    potential is that of G = 1 and shift = 50, scaled."""
    nx, ny, nz = shape
    rho = np.random.default_rng(6).integers(0, 2 ** 45, size=(nz, ny, nx))
    a = _static(rho, shape)
    k = G + 50 - shift   # the power of two between the two
    b = _static(rho, shape, shift=shift, G=2.0 ** G)
    assert b.any()
    # Every conversion's unit is at most 2^-1018 where a group lies that low: of
    # H-hat (times the sum of masses, for each of the 8N modes), of the masses'
    # spectra (times the sum of H-hat, 8N H(0), H(0) below 4N G) and of the
    # potential's (8N values summed twice)
    N8, M, g = 8.0 * rho.size, float(rho.sum()) * 2.0 ** -shift, 2.0 ** G
    unit = N8 * (M + 4 * g * N8 + 2) * 2.0 ** -1018
    tol = unit + 64 * 2.0 ** -53 * np.ldexp(np.abs(a).max(), k)
    print(f"tolerance {tol / np.ldexp(np.abs(a).max(), k):.1e} of the largest value")
    assert np.abs(b - np.ldexp(a, k)).max() <= tol


@pytest.mark.parametrize("shape", [(16, 16, 16), (64, 32, 32), (8, 64, 16)])
@pytest.mark.parametrize("G", [0.0, -0.0, 2.0 ** -1060, -2.0 ** -1060])
def test_vanishing_strength(shape, G):
    """No Green's function, and one whose potential is below every FP64 number:
    groups of zeros of either sign stay zero."""
    nx, ny, nz = shape
    rho = np.random.default_rng(6).integers(-2 ** 45, 2 ** 45, size=(nz, ny, nx))
    b = _static(rho, shape, G=G)
    if G == 0:
        assert not b.any()
    # the unit of the conversions (see test_small_magnitudes)
    N8, M = 8.0 * rho.size, float(np.abs(rho).sum()) * 2.0 ** -50
    assert np.abs(b).max() <= N8 * (M + 2) * 2.0 ** -1018
