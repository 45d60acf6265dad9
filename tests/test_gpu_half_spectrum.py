"""A single real mass set is transformed by its half spectrum: two rows a
complex row in the x passes, the columns kx <= nx in the others.  Shapes where
the half rounds up to whole tiles, fills them exactly or is no less than the
whole (short rows), alone and as the odd item of a batch of two systems'
shapes, against the oracle."""
import math

import numpy as np
import pytest

import oracle as O
from tests._harness import gpu_setup
from tests.test_zz_no_alloc import _single_grid

pytestmark = pytest.mark.gpu


def _check(w, shape, key, ctx):
    rho, phi = ctx.density(*key), ctx.potential(*key).astype(np.float64)
    s = w["system"]
    g = ctx.gals[key[0]].coarse
    geo = O.geometry_from_spec(w["galaxies"][key[0]]["coarse"])
    assert (g.nx, g.ny, g.nz) == shape and np.count_nonzero(rho) > 20   # 8^3: the points fill 27 cells
    ref = O.potential_fft(O.rho_real(rho, ctx.info()["shift"]), geo, s["G"], s["h000"])
    # forward and inverse transform of N points: at most eps log2 N each in the 2-norm
    n = 8 * shape[0] * shape[1] * shape[2]
    tol = 2 * math.log2(n) * (2.0 ** -24 if w["precision"] == "fp32" else 2.0 ** -53)
    assert np.linalg.norm(phi - ref) <= tol * np.linalg.norm(ref)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("shape", [
    (8, 8, 8), (8, 256, 8), (256, 8, 8), (16, 16, 64), (64, 16, 16), (16, 64, 256), (128, 32, 8), (32, 128, 128),
    (64, 256, 32), (256, 64, 16)])
def test_half_spectrum_shapes(shape, precision):
    w = _single_grid(*shape, 1.0, precision)
    ctx, parts = gpu_setup(w)
    ctx.deposit(parts)
    ctx.solve()
    _check(w, shape, (0, 5), ctx)
    ctx.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("batched", [0, 1])
def test_half_spectrum_batches(precision, batched):
    """Two galaxies of one single-grid shape and one of another."""
    shapes = [(32, 16, 16), (32, 16, 16), (64, 32, 8)]
    ws = [_single_grid(*s, 1.0, precision, n=3000, seed=i) for i, s in enumerate(shapes)]
    w = dict(ws[0], galaxies=[dict(x["galaxies"][0]) for x in ws],
             pos=np.concatenate([x["pos"] for x in ws], 1), vel=np.concatenate([x["vel"] for x in ws], 1),
             m=np.concatenate([x["m"] for x in ws]), gal=np.repeat(np.arange(3, dtype=np.int32), 3000))
    ctx, parts = gpu_setup(w)
    ctx.set_launch_config(batched, 0)
    ctx.deposit(parts)
    ctx.solve()
    for g, s in enumerate(shapes):
        _check(w, s, (g, 5), ctx)
    ctx.close()
