"""Steps past t_end leave the state as it is, an odd number of them too, in the steps that change buffers: the
semi-Lagrangian ones and the fused D2Q16 one (the fused D1Q4 one: test_gpu_chunk.py)."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,nx,ny,scheme,fused", [(1, 300, 1, "sl", 0), (2, 37, 21, "sl", 0), (2, 37, 21, "fv", 1), (2, 9, 40, "fv", 2)])
def test_past_t_end(dim, nx, ny, scheme, fused, precision):
    pb = I.smooth_periodic(dim, nx, ny, seed=5, amp=0.15)
    kw = dict(precision=precision, tau=1e-5, cfl=0.2, scheme=scheme)
    s = pond.Solver(pb, **kw)
    s.set_variants(0, 0, fused)
    s.set_primitive()
    s.step(20)
    t = s.sync()["t"]
    s.close()
    e = pond.Solver(pb, t_end=0.9 * t, **kw)
    e.set_variants(0, 0, fused)
    e.set_primitive()
    for n in range(30):   # to t_end and past it, launch by launch
        e.step(1)
        if e.sync()["dt"] == 0.0:
            break
    d = e.sync()
    assert d["dt"] == 0.0 and d["t"] == pytest.approx(0.9 * t)
    read = lambda: [*e.state(), *([] if scheme == "sl" else e.face_gauges())]
    want = read()
    for n in (1, 1, 2, 3, 33, 32):
        e.step(n)
        for a, b in zip(read(), want):
            assert np.array_equal(a, b)
    assert e.sync()["steps"] == d["steps"]
    e.close()
