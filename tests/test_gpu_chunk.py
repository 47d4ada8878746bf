"""The fused D1Q4 step (a warp per chunk of cells, one or four lanes per face) against the oracle at the
edges of its chunks under every ghost rule, past t_end, and through graphs entered on either set of
planes.

FP64 tolerance: a step carries a few hundred roundings of 1e-16, the corrector stops at 1e-13, and
inputs perturbed by 1e-15 move the oracle by at most TOL / 100 on these flows."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import max_rel, oracle_for, rel_l1  # noqa: E402
from tests.test_gpu_parity import gpu_for  # noqa: E402

pytestmark = pytest.mark.gpu

TOL = 1e-11
BCS = {"open": (0, 0), "periodic": (1, 1), "inflow_wall": (2, 3), "wall_inflow": (3, 2)}


def tube(n, bc):
    pb = I.shock_tube((1.0, 0.3, 1.0), (0.5, -0.2, 0.6), 1.4, n)
    pb.rho = pb.rho * (1.0 + 0.05 * np.sin(7.0 * I.cell_centres(n, 0.0, 1.0)))
    pb.bc = bc + (0, 0)
    for side in range(2):
        if bc[side] == 2:
            pb.inflow[side] = (0.9, 0.1, 0.0, 0.8)
            pb.inflow_range[side] = (0, 1)
    return pb


@pytest.mark.parametrize("n", [1, 2, 3, 6, 7, 8, 13, 14, 27, 28, 29, 30, 57, 113])
@pytest.mark.parametrize("bc", sorted(BCS))
def test_chunk_edges(n, bc):
    pb = tube(n, BCS[bc])
    kw = dict(tau=1e-5, cfl=0.2, tol=1e-13, max_iter=10)
    o = oracle_for(pb, **kw)
    o.step(5)
    st = o.stats()
    for prec in ("fp64", "fp32"):
        s = gpu_for(pb, precision=prec, **kw)
        for v in (1, 2):
            s.set_variants(0, 0, v)
            s.set_primitive()
            s.step(5)
            d = s.sync()
            assert d["face_solves"] == 5 * (n + 1) and d["steps"] == 5 and d["fallbacks"] == st["fallbacks"]
            got, want = s.moments(totals=False)[0], o.conserved()
            if prec == "fp64":
                for k in (0, 1, 3):
                    assert max_rel(got[k], want[k]) <= TOL, (v, k)
                assert max_rel(s.face_gauges()[0], o.face_gauges()[0]) <= TOL
            else:
                for k in (0, 3):
                    assert rel_l1(got[k], want[k]) <= 1e-4, (v, k)
        s.close()


@pytest.mark.parametrize("variant", [0, 1, 2])
def test_past_t_end_and_graphs(variant):
    """Steps after t_end leave the state as it is, an odd number of them too (the fused step changes
    buffers); runs of graphs entered on either set of planes equal single launches."""
    pb = tube(61, (0, 0))
    kw = dict(tau=1e-5, cfl=0.2, max_iter=8)
    a, b = (gpu_for(pb, precision="fp64", **kw) for _ in range(2))
    for s in (a, b):
        s.set_variants(0, 0, variant)
        s.set_primitive()
    for n in (1, 64, 33, 32):
        a.step(n)
    for _ in range(130):
        b.step(1)
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    t = a.sync()["t"]
    e = gpu_for(pb, precision="fp64", t_end=0.7 * t, **kw)
    e.set_variants(0, 0, variant)
    e.set_primitive()
    e.step(110)
    at_end, gauges, d = e.state(), e.face_gauges()[0], e.sync()
    assert d["t"] == pytest.approx(0.7 * t) and d["steps"] < 110
    e.step(1)
    for x, y in zip(e.state(), at_end):
        assert np.array_equal(x, y)
    e.step(34)
    for x, y in zip(e.state(), at_end):
        assert np.array_equal(x, y)
    assert np.array_equal(e.face_gauges()[0], gauges)
