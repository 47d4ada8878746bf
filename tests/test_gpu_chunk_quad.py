"""The D1Q4 FP64 step with four lanes per face, where the corrector's stop hangs on the last bits: with the
tolerance at a few roundings each pass either just meets it or just does not, and the four lanes of a face have
to decide alike (they exchange in the next pass).

Bound: a step carries a few hundred roundings of 1e-16, and a corrector stopped a pass early or late
moves its frame by the tolerance, 40 steps at 2e-15 and below: 1e-11 leaves a decade, as for the other
D1Q4 tests."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import max_rel, oracle_for  # noqa: E402
from tests.test_gpu_parity import gpu_for  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tol", [2e-16, 4e-16, 1e-15, 2e-15])
@pytest.mark.parametrize("n", [5, 7, 8, 200, 1001])
def test_stop_at_rounding(n, tol):
    pb = I.shock_tube((1.0, 0.3, 1.0), (0.5, -0.2, 0.6), 1.4, n)
    pb.rho = pb.rho * (1.0 + 0.05 * np.sin(7.0 * I.cell_centres(n, 0.0, 1.0)))
    kw = dict(tau=1e-5, cfl=0.2, tol=tol, max_iter=12)
    o = oracle_for(pb, **kw)
    o.step(40)
    runs = []
    for _ in range(2):
        s = gpu_for(pb, precision="fp64", **kw)
        s.set_variants(0, 0, 2)
        s.set_primitive()
        s.step(40)
        d = s.sync()
        assert d["steps"] == 40 and d["face_solves"] == 40 * (n + 1)
        got = s.moments(totals=False)[0]
        for k in (0, 1, 3):
            assert max_rel(got[k], o.conserved()[k]) <= 1e-11
        runs.append((d["face_iters"], *s.state()))
        s.close()
    assert runs[0][0] == runs[1][0]   # the same passes, and the same bits, each time
    for a, b in zip(runs[0][1:], runs[1][1:]):
        assert np.array_equal(a, b)
