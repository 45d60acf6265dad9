"""Contexts made and used by several threads at once: the launch sizes that
are found once per process and kept."""
import threading

import numpy as np
import pytest

from paper_1210_1736_gb300 import pm, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_threads_make_contexts_together(precision):
    import torch
    w = W.galaxy_small(precision=precision, n_total=4000)
    dt = torch.float32 if precision == "fp32" else torch.float64
    out, err, go = [None] * 5, [], threading.Barrier(4)

    def work(k):
        try:
            if k < 4:
                go.wait(60)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                ctx = pm.Context(w, W.mass_bound(w["m"]))
                p = pm.Particles(w["pos"], w["vel"], w["m"], w["gal"], precision=precision)
                assert p.dtype == dt
                ctx.recentre(p)
                ctx.deposit(p)
                ctx.solve()
                out[k] = {key: ctx.potential(*key) for key in ctx.shapes}
                ctx.close()
        except Exception as e:   # reported by the main thread
            err.append(e)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    work(4)
    assert not err, err
    for k in range(4):
        for key in out[4]:
            assert np.array_equal(out[k][key], out[4][key]), (k, key)
