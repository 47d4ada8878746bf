"""Face variant indices of D2Q16 grids past the end of the present list: those of the longest list are taken still
and run the variant that the grid starts on (the same bits), the next one is refused as ever."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,most", [("fp32", 14), ("fp64", 4)])
def test_indices_of_the_longest_list(precision, most):
    pb = I.quadrants_2d(37, seed=1)
    s = pond.Solver(pb, precision=precision, tau=1e-5, cfl=0.2)
    present = sum(1 for n in s.variants() if n.startswith("face "))
    out = []
    for face in [None] + list(range(present, most)):
        if face is not None:
            s.set_variants(face=face)
        s.set_primitive()
        s.step(4)
        assert s.sync(raise_on_error=False)["steps"] == 4
        out.append(s.state())
    assert len(out) > 1
    for got in out[1:]:
        for a, b in zip(got, out[0]):
            assert np.array_equal(a, b, equal_nan=True)   # (this draw has cells without a state)
    for bad in (-1, most):
        with pytest.raises(pond.PondError):
            s.set_variants(face=bad)
    s.close()
