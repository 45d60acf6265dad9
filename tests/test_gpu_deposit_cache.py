"""The unsorted deposit's block cache: densities are exact whatever shares a
slot, fills the table or sits in one cell."""
import numpy as np
import pytest

import oracle as O
from paper_1210_1736_gb300 import workloads as W
from tests._harness import gpu_setup, oracle_setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,how", [(1, "spread"), (255, "one cell"), (4_097, "one cell"), (60_000, "uniform"),
                                   (300_000, "spread"), (700_001, "one cell")])
def test_exact(precision, n, how):
    w = W.galaxy_small(precision=precision, n_total=max(n, 100))
    for k in ("pos", "vel"):
        w[k] = w[k][:, :n].copy()
    w["m"], w["gal"] = w["m"][:n].copy(), w["gal"][:n]
    rng = np.random.default_rng(n)
    if how == "one cell":
        w["pos"][:] = rng.uniform(-0.01, 0.01, w["pos"].shape)
    elif how == "uniform":   # every coarse cell: more cells than the table has slots
        w["pos"][:] = rng.uniform(-18, 18, w["pos"].shape)
    # masses whose sums carry from the low word, both signs
    w["m"] *= rng.choice([1.0, -1.0, 2.0 ** -20], n)
    ctx, parts = gpu_setup(w)
    ctx.deposit(parts)
    system, state = oracle_setup(w)
    flags, own = O.classify(state, system)
    rho, flags, _ = O.deposit(state, system, flags, own)
    for k, ref in rho[0].items():
        assert np.array_equal(ctx.density(0, k), ref), k
