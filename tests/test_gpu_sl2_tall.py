"""D2Q16 semi-Lagrangian grids of more rows than 65 535 tiles hold: a field that repeats along y gives the same
rows as one period of it with periodic sides.

Bound: both take the same steps on the same values; only the tiles' reference velocities differ (FP64: a
few roundings a step, 1e-13; FP32: offsets of order one rounded to 6e-8, some ten a step)."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import max_rel  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bound", [("fp64", 1e-13), ("fp32", 4e-6)])
def test_more_tile_rows_than_a_grid_dimension(precision, bound):
    nx, period, times = 5, 24, 5470   # 131 280 rows
    pb = I.smooth_periodic(2, nx, period, seed=2, amp=0.1)
    rows = lambda a: np.tile(np.asarray(a).reshape(period, nx), (times, 1)).ravel()
    tall = I.Problem(2, nx, period * times, pb.x0, pb.x1, pb.y0, pb.y0 + times * (pb.y1 - pb.y0), pb.gamma, rows(pb.rho), rows(pb.ux),
                     rows(pb.uy), rows(pb.p), bc=pb.bc)
    got = []
    for q in (pb, tall):
        s = pond.Solver(q, precision=precision, tau=1e-5, cfl=0.2, scheme="sl", fixed_iters=3, max_iter=8)
        s.set_primitive()
        s.step(3)
        assert s.sync()["nonphysical"] == 0
        got.append([np.asarray(a) for a in s.moments(totals=False)[0]])
        s.close()
    for a, b in zip(*got):
        assert max_rel(b, rows(a)) <= bound
