"""A semi-Lagrangian solver that is set again after any number of steps gives the bits of a new one: its steps swap the
state with the face planes, which setting the fields must not take for faces then."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("dim,nx,ny", [(1, 200, 1), (1, 1001, 1), (2, 45, 119), (2, 16, 8)])
def test_set_again(dim, nx, ny, precision):
    pb = I.smooth_periodic(dim, nx, ny, seed=5, amp=0.15)
    kw = dict(precision=precision, tau=1e-5, cfl=0.2, scheme="sl")
    s, want = pond.Solver(pb, **kw), None
    for before in (0, 1, 2, 33, 3):
        if before:
            s.step(before)
        s.set_primitive()
        s.step(7)
        d = s.sync()
        assert d["steps"] == 7
        got = [*s.state(), *s.moments(totals=False)[0]]
        if want is None:
            want = got
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
    s.close()
