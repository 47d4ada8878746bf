"""The D2Q16 lane face kernel (two faces a thread in FP32, unfinished faces worked off by 16 lanes
each) against the oracle where it can go wrong: grids below, at and above a tile in either
direction, single rows and columns, every ghost rule, converging and fixed-count correctors, and
faces whose passes define no frame.

FP64 tolerance: both sides evaluate the same expressions in FP64 with other associations; a step
carries a few hundred roundings of 1e-16, the corrector stops at 1e-13, and inputs perturbed by
1e-15 move the oracle's results by at most 4e-14 on these draws, so 1e-11 of the largest value
leaves two decades."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import max_rel, oracle_for, rel_l1  # noqa: E402
from tests.test_gpu_parity import gpu_for  # noqa: E402

pytestmark = pytest.mark.gpu


def crop(pb, nx, ny):
    """The middle nx x ny cells of a square problem (its ghost rules and cell size kept)."""
    n = pb.nx
    i, j = (n - nx) // 2, (n - ny) // 2
    cut = lambda a: np.ascontiguousarray(np.asarray(a).reshape(n, n)[j:j + ny, i:i + nx]).ravel()
    return I.Problem(2, nx, ny, 0.0, nx * pb.dx, 0.0, ny * pb.dy, pb.gamma, cut(pb.rho), cut(pb.ux), cut(pb.uy), cut(pb.p),
                     bc=pb.bc)


def run(pb, variant, precision, steps, limiter, **kw):
    s = gpu_for(pb, precision=precision, limiter=limiter, **kw)
    s.set_variants(face=variant)
    s.set_primitive()
    s.step(steps)
    d = s.sync()
    out, _ = s.moments(totals=False)
    s.close()
    return out, d


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (9, 1), (7, 3), (8, 4), (15, 8), (16, 8), (17, 9), (33, 5), (32, 33)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 3, 3), (3, 0, 1, 1)], ids=["open", "periodic_x_walls_y", "wall_x_periodic_y"])
def test_tile_edges(nx, ny, bc):
    pb = crop(I.quadrants_2d(34, seed=3, mach_max=0.4), nx, ny)
    pb.bc = bc
    kw = dict(tau=1e-5, cfl=0.2, tol=1e-13, max_iter=12)
    o = oracle_for(pb, limiter=1, **kw)
    o.step(3)
    for v in range(3):
        got, d = run(pb, v, "fp64", 3, 1, **kw)
        assert d["face_solves"] == 3 * ((nx + 1) * ny + nx * (ny + 1))
        for a, b in zip(got, o.conserved()):
            assert max_rel(a, b) <= 1e-11, v
        got, d = run(pb, v, "fp32", 3, 1, **kw)
        assert d["face_solves"] == 3 * ((nx + 1) * ny + nx * (ny + 1))
        for k in (0, 3):   # density and energy (momentum may vanish between walls)
            assert rel_l1(got[k], o.conserved()[k]) <= 1e-4, v


@pytest.mark.parametrize("fixed", [0, 1, 4])
def test_faces_without_a_frame(fixed):
    """A draw whose corrector meets passes without a frame (restarts, stops at the last valid
    pass): the counts of passes, restarts and faces at the limit are the oracle's too."""
    pb = I.quadrants_2d(40, seed=0, direction="any")
    kw = dict(tau=1e-5, cfl=0.2, max_iter=9, fixed_iters=fixed, tol=1e-12)
    o = oracle_for(pb, **kw)
    o.step(2)
    st = o.stats()
    got, d = run(pb, 0, "fp64", 2, 0, **kw)
    assert d["fallbacks"] == st["fallbacks"] and d["face_iters"] == st["face_iters"]
    for a, b in zip(got, o.conserved()):
        assert max_rel(a, b) <= 1e-11
