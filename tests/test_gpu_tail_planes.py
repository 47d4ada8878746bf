"""The grid-wide tail's list lies in the planes of the learned predictions.  A learned step after plain ones must not
depend on what the list left there: FP64 grids of many faces along x and few along y, with a tolerance at
which faces stop apart and warps hand over what is left, for a long list.  Which words it leaves differs from run to run (faces take their places in the order of
atomics) and with what ran before, so runs after different pasts have to give the same bits."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def params():
    rng = np.random.default_rng(4)
    p = rng.normal(0.0, 0.15, pond.MLP_PARAMS).astype(np.float32)
    return p


@pytest.mark.parametrize("precision,tol", [("fp64", 3e-16), ("fp32", 1e-7)])
def test_learned_steps_do_not_see_the_list(precision, tol):
    pb = I.smooth_periodic(2, 700, 6, seed=3, amp=0.15)
    other = I.quadrants_2d(700, seed=2)
    past = [np.asarray(f).reshape(700, 700)[300:306].ravel().copy() for f in (other.rho, other.ux, other.uy, other.p)]
    runs = []
    for before in (0, 0, 5):
        s = pond.Solver(pb, precision=precision, tau=1e-5, cfl=0.2, tol=tol, max_iter=12)
        s.set_gauge_params(params())
        if before:   # another flow's list first
            s.set_primitive(*past)
            s.step(before)
            s.sync(raise_on_error=False)
        s.set_primitive(pb.rho, pb.ux, pb.uy, pb.p)
        s.step(3)
        s.gauge_enable(True)
        s.step(4)
        s.gauge_enable(False)
        s.step(2)
        s.gauge_enable(True)
        s.step(3)
        d = s.sync(raise_on_error=False)
        runs.append(({k: d[k] for k in ("steps", "face_iters", "nonconverged", "fallbacks", "t", "dt")}, *s.state(), *s.face_gauges()))
        s.close()
    for r in runs[1:]:
        np.testing.assert_equal(r[0], runs[0][0])
        for a, b in zip(r[1:], runs[0][1:]):
            assert np.array_equal(a, b, equal_nan=True)
