"""The D3Q64 face kernel and its tail against the oracle where they can go wrong: boxes below, at and
above a tile along each axis, single layers, every ghost rule, converging correctors (every
unfinished face goes through the list on grids of this size in FP64) and passes without a frame.

FP64 tolerance: other associations of the same expressions, a few thousand roundings of 1e-16 a
step, correctors stopped at 1e-13; inputs perturbed by 1e-15 move the oracle by up to 8e-13 on the
first test's flows and 8e-15 on the second's, so 1e-10 and 1e-12 leave two decades."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import max_rel, oracle_for, rel_l1  # noqa: E402

pytestmark = pytest.mark.gpu


def crop3(pb, nx, ny, nz, bc):
    """The middle nx x ny x nz cells of a cubic problem."""
    n = pb.nx
    i, j, k = (n - nx) // 2, (n - ny) // 2, (n - nz) // 2
    cut = lambda a: np.ascontiguousarray(np.asarray(a).reshape(n, n, n)[k:k + nz, j:j + ny, i:i + nx]).ravel()
    return I.Problem3(nx, ny, nz, 0, nx * pb.dx, 0, ny * pb.dy, 0, nz * pb.dz, pb.gamma, cut(pb.rho), cut(pb.ux), cut(pb.uy),
                      cut(pb.uz), cut(pb.p), bc=bc)


def run(pb, variant, precision, steps, **kw):
    s = pond.Solver3(pb, precision=precision, **kw)
    s.set_variants(face=variant)
    s.set_primitive()
    s.step(steps)
    d = s.sync()
    out, _ = s.moments(totals=False)
    s.close()
    return out, d


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (1, 5, 3), (4, 4, 2), (5, 3, 4), (9, 4, 1), (8, 5, 5)])
@pytest.mark.parametrize("bc", [(0,) * 6, (1, 1, 3, 3, 0, 3)], ids=["open", "mixed"])
def test_tile_edges_3d(nx, ny, nz, bc):
    pb = crop3(I.octants_3d(10, seed=3, mach_max=0.4), nx, ny, nz, bc)
    kw = dict(tau=1e-5, cfl=0.2, tol=1e-13, max_iter=10)
    faces = (nx + 1) * ny * nz + nx * (ny + 1) * nz + nx * ny * (nz + 1)
    o = oracle_for(pb, **kw)
    o.step(2)
    for v in range(3):
        got, d = run(pb, v, "fp64", 2, **kw)
        assert d["face_solves"] == 2 * faces
        for a, b in zip(got, o.conserved()):
            assert max_rel(a, b) <= 1e-10, v
        got, d = run(pb, v, "fp32", 2, **kw)
        assert d["face_solves"] == 2 * faces
        for k in (0, 4):   # density and energy (momentum may vanish between walls)
            assert rel_l1(got[k], o.conserved()[k]) <= 1e-4, v


@pytest.mark.parametrize("fixed", [0, 3])
def test_passes_without_a_frame_3d(fixed):
    """Restarts and stops at the last valid pass, counted as the oracle counts them."""
    pb = I.octants_3d(8, seed=3, mach_max=4.0)
    kw = dict(tau=1e-5, cfl=0.2, max_iter=7, fixed_iters=fixed, tol=1e-12)
    o = oracle_for(pb, **kw)
    o.step(1)
    st = o.stats()
    assert st["fallbacks"] > 0
    got, d = run(pb, 0, "fp64", 1, **kw)
    assert d["fallbacks"] == st["fallbacks"] and d["face_iters"] == st["face_iters"]
    for a, b in zip(got, o.conserved()):
        assert max_rel(a, b) <= 1e-12

