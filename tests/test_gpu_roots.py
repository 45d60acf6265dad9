"""The FP64 roots from an FP32 seed (pm_roots.cuh) against extended precision:
over the seed's exponent range, at both fall-back limits and beyond them."""
import numpy as np
import pytest

from paper_1210_1736_gb300 import pm

pytestmark = pytest.mark.gpu


def _roots(r):
    import torch
    t = torch.tensor(r, device="cuda")
    out = [torch.empty_like(t) for _ in range(3)]
    pm._check(pm.lib().pm_selftest_roots(t.data_ptr(), len(r), *[o.data_ptr() for o in out],
                                         torch.cuda.current_stream().cuda_stream))
    return [o.cpu().numpy() for o in out]


def _arguments(kind):
    rng = np.random.default_rng(8)
    if kind == "squares":   # squared distances of cells, the arguments of H
        i, j, k = rng.integers(0, 257, size=(3, 200_000))
        q = rng.choice([1.0, 0.25, 0.8, 1 / 3], size=len(i))
        r = (i * i + j * j).astype(np.float64) + (q * k) ** 2
        return r[r > 0]
    if kind == "range":
        return 2.0 ** rng.uniform(-99.6, 99.6, size=400_000)
    if kind == "limits":   # both sides of the fall-back limits (also as FP32 sees them)
        out = []
        for x in (1e-30, 1e30, float(np.float32(1e-30)), float(np.float32(1e30))):
            for d in range(-40, 41):
                out += [x * (1 + d * 2.0 ** -52), x * (1 + d * 2.0 ** -24)]
        return np.array(out)
    return np.concatenate([2.0 ** rng.uniform(100, 1023, size=20_000), 2.0 ** rng.uniform(-1021, -100, size=20_000),
                           [5e-324, 2.0 ** -1022, 1.7e308]])


@pytest.mark.parametrize("kind", ["squares", "range", "limits", "beyond"])
def test_roots(kind):
    r = _arguments(kind)
    inv_sqrt, root, inv = _roots(r)
    x = np.sqrt(r.astype(np.longdouble))
    # 1.5 x 2^-53 by the seed's step (see pm_roots.cuh), 2^-52 by the quotient of
    # a rounded root; the long doubles' rounding and the step's rest are below 2^-60
    bound = 2.0 ** -52 if kind in ("limits", "beyond") else 1.5 * 2.0 ** -53
    for v in (inv_sqrt, inv):
        assert np.abs(v * x - 1).max() <= bound + 2.0 ** -60
    assert np.abs(root / x - 1).max() <= 2.0 ** -53 + 2.0 ** -60
    assert np.array_equal(root, np.sqrt(r))   # none of these arguments is a near tie


def test_zero_and_infinity():
    inv_sqrt, root, inv = _roots(np.array([0.0, np.inf]))
    assert np.array_equal(inv_sqrt, [np.inf, 0.0]) and np.array_equal(root, [0.0, np.inf]) and np.array_equal(inv, [0.0, 0.0])
