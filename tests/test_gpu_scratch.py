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
