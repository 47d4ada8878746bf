"""The D2Q16 semi-Lagrangian kernel where a node's stop hangs on the last bits: four lanes work on a node, each
going on or stopping by its own copy of the moments, so the copies must be the same bits.

Bounds: 1e-12 in FP64, as in the other parity tests of this kernel (a corrector that stops a pass early or late
moves its frame by the tolerance, 2e-15 at most).  FP32: three steps of up to eight passes, each some
forty dependent roundings of 2^-24 on values of order one: 24 * 40 * 6e-8 = 6e-5 if they all added up."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import rel_l1  # noqa: E402
from tests.test_gpu_parity import compare_fp64  # noqa: E402
from tests.test_gpu_sl import sl_pair  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [("fp64", 2e-16), ("fp64", 2e-15), ("fp32", 6e-8), ("fp32", 2e-7)])
@pytest.mark.parametrize("nx,ny", [(9, 3), (33, 25), (64, 48)])
def test_stop_at_rounding(nx, ny, precision, tol):
    pb = I.smooth_periodic(2, nx, ny, seed=nx, amp=0.15)
    kw = dict(tau=1e-5, tol=tol, max_iter=8)
    bits = []
    for _ in range(2):
        gs, os_ = sl_pair(pb, 0.2, precision=precision, **kw)
        gs.step(3)
        os_.sl_step(3)
        d = gs.sync()
        assert d["nonphysical"] == 0 and d["steps"] == 3
        if precision == "fp64":
            compare_fp64(gs, os_, tol=1e-12, faces=False)
        else:
            (r, _, _, E), _ = gs.moments(totals=False)
            ro, _, _, Eo = os_.conserved()
            assert rel_l1(r, ro) <= 6e-5 and rel_l1(E, Eo) <= 6e-5
        bits.append((np.array(d["face_iters"]), *gs.state()))
        gs.close()
    for a, b in zip(*bits):
        assert np.array_equal(a, b)
