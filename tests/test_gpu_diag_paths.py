"""Disc diagnostics: each accumulator layout (a column per thread of 64 or 32
threads, one set per block), one bin, as many boundaries as there are
counters' rows, and selections of a few particles."""
import numpy as np
import pytest

from oracle import pm_diag as D
from paper_1210_1736_gb300 import workloads as W
from tests._harness import gpu_setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nbins,nring,mmax,nsel", [(1, 1, 1, None), (20, 10, 4, None), (33, 3, 7, 100),
                                                   (64, 10, 4, None), (64, 16, 64, 5000), (64, 1, 1, 3), (5, 4, 2, 0)])
def test_layouts(precision, nbins, nring, mmax, nsel):
    import torch
    w = W.galaxy_small(precision=precision, n_total=20_000)
    ctx, parts = gpu_setup(w)
    ctx.deposit(parts)
    disc = np.asarray(w["comp"]) == W.COMP_DISC
    if nsel is not None:
        disc &= np.cumsum(disc) <= nsel
    for _ in range(2):   # the scratch is left as the next call wants it
        got = ctx.disc_diagnostics(parts, torch.tensor(disc, device="cuda"), nbins=nbins, nring=nring, mmax=mmax)["raw"]
    if not disc.any():
        assert not got.any()
        return
    pos, vel, flags = parts.host()
    ref = D.disc_diagnostics(pos, vel, parts.m.cpu().numpy().astype(np.float64), disc, (flags & 1) == 0,
                             ctx.centres()[0], nbins, nring, mmax, 5.0, 3.2, 0.4)
    counts = slice(7, 6 + 4 * nbins, 4)
    assert np.array_equal(got[counts], ref[counts]) and got[0] == ref[0]
    # FP64 sums of at most 20,000 terms in another order: 2e4 * 2^-53 of the
    # summed magnitudes, which the smallest modes are about 1e-3 of
    tol = 1e-9 * np.abs(ref) + 1e-12 * np.abs(ref[6 + 4 * nbins:]).max(initial=0.0)
    assert np.all(np.abs(got - ref) <= tol)
