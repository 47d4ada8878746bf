"""FP32 D1Q4 steps round alike in the fused kernel and in the face and cell kernels: a shocked FP32 tube amplifies
a change of rounding (limiters switch, correctors cycle) by orders of magnitude, so nothing but equal
bits says that a variant solves the same flow.  Sizes at the edges of chunks (28 cells) and of the blocks of 128 faces
that share a reference velocity, every ghost rule, both limiters, and states whose correctors restart."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def outputs(pb, variant, steps, **kw):
    s = pond.Solver(pb, precision="fp32", tau=1e-5, **kw)
    if variant is not None:
        s.set_variants(0, 0, variant)
    s.set_primitive()
    s.step(steps)
    d = s.sync(raise_on_error=False)
    out = [*s.state(), s.face_gauges()[0]]
    s.close()
    return out, {k: d[k] for k in ("t", "dt", "steps", "face_solves", "face_iters", "nonconverged", "fallbacks")}


def same_bits(pb, steps, **kw):
    want, dw = outputs(pb, 0, steps, **kw)
    for v in (1, 2, None):
        got, dg = outputs(pb, v, steps, **kw)
        np.testing.assert_equal(dg, dw)
        for a, b in zip(got, want):
            assert np.array_equal(a, b, equal_nan=True), v
    return dw


@pytest.mark.parametrize("n", [1, 2, 27, 28, 29, 127, 128, 129, 140, 255, 256, 257, 1000])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1), (2, 3), (3, 2)], ids=["open", "periodic", "inflow_wall", "wall_inflow"])
def test_edges(n, bc):
    rng = np.random.default_rng(n)
    pb = I.shock_tube((1.0, 0.75, 1.0), (0.125, 0.0, 0.1), 1.4, n)
    pb.rho = pb.rho * (1.0 + 0.2 * rng.uniform(-1.0, 1.0, n))
    pb.bc = bc + (0, 0)
    for side in range(2):
        if bc[side] == 2:
            pb.inflow[side] = (0.9, 0.1, 0.0, 0.8)
            pb.inflow_range[side] = (0, 1)
    same_bits(pb, 37, cfl=0.3, limiter=n % 2)


def test_restarts_and_stops():
    """Random strong tubes: some correctors meet passes without a frame (restart, stop at the last valid
    pass, none at all), some stop at the limit."""
    rng = np.random.default_rng(7)
    fallbacks = 0
    for k in range(24):
        n = int(rng.integers(20, 400))
        e, u = rng.uniform(-5.0, 5.0, (2, 2)), rng.uniform(-8.0, 8.0, 2)
        pb = I.shock_tube((np.exp(e[0, 0]), u[0], np.exp(e[0, 1])), (np.exp(e[1, 0]), u[1], np.exp(e[1, 1])), 1.4, n)
        fallbacks += same_bits(pb, 1 + k, cfl=0.5, limiter=k % 2, max_iter=(1, 2, 5, 16)[k % 4], fixed_iters=3 * (k % 6 == 5))["fallbacks"]
    assert fallbacks > 0
