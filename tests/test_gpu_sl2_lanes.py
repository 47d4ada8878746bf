"""The D2Q16 semi-Lagrangian kernel at the edges of its tiles (8 x 8 nodes in FP32, 8 x 2 in FP64, four
lanes a node, eight nodes a warp): grids smaller than a warp's nodes, of exactly a tile, one past
it, and ragged in both directions, with walls and with periodic sides."""
import pytest

torch = pytest.importorskip("torch")

from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import rel_l1  # noqa: E402
from tests.test_gpu_parity import compare_fp64  # noqa: E402
from tests.test_gpu_sl import KW64, sl_pair  # noqa: E402
from tests.test_oracle_reflective import perturbed, walled  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(3, 2), (8, 2), (9, 3), (7, 17), (16, 8), (17, 9)]


def problem(nx, ny, walls):
    pb = I.smooth_periodic(2, nx, ny, seed=nx + ny, amp=0.1)
    return walled(perturbed(pb, 3)) if walls else pb


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("walls", [False, True])
def test_tiles_fp64(nx, ny, walls):
    """The bound of the other FP64 parity tests: 1e-12."""
    gs, os_ = sl_pair(problem(nx, ny, walls), 0.2, **KW64)
    gs.step(3)
    os_.sl_step(3)
    d, st = gs.sync(), os_.stats()
    assert d["face_iters"] == st["face_iters"] and d["nonphysical"] == st["nonphysical"] == 0
    compare_fp64(gs, os_, tol=1e-12, faces=False)


@pytest.mark.parametrize("nx,ny", SIZES + [(8, 8), (33, 25)])
def test_tiles_fp32(nx, ny):
    """Three steps of three passes, each some forty dependent roundings of 2^-24 on values of order
    one: 9 * 40 * 6e-8 = 2e-5 if they all added up."""
    gs, os_ = sl_pair(problem(nx, ny, True), 0.2, precision="fp32", **KW64)
    gs.step(3)
    os_.sl_step(3)
    (r, _, _, E), _ = gs.moments(totals=False)
    ro, _, _, Eo = os_.conserved()
    assert rel_l1(r, ro) <= 2e-5 and rel_l1(E, Eo) <= 2e-5
