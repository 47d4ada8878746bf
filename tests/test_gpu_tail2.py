"""The grid-wide tail of the D2Q16 lane kernel: its list lies in the planes of the learned predictions, so
steps without the predictor must leave nothing there that a later learned step takes for one; and
the default face variant on both sides of the size at which it changes.

FP32 tolerance: 1e-5 relative L1, the bound at which the tile variants are held to each other."""
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402
from tests.common import rel_l1  # noqa: E402

pytestmark = pytest.mark.gpu


def fields(pb, variant=None, learned_after=None, steps=4):
    s = pond.Solver(pb, precision="fp32", tau=1e-5, cfl=0.2, tol=1e-6)
    if variant is not None:
        s.set_variants(face=variant)
    s.set_primitive()
    if learned_after is not None:
        s.step(learned_after)
        s.gauge_enable(True)
    s.step(steps)
    d = s.sync()
    assert d["nonphysical"] == 0
    out, _ = s.moments(totals=False)
    s.close()
    return out, d


@pytest.mark.parametrize("nx,ny", [(37, 21), (64, 40)])
def test_learned_steps_after_plain_ones(nx, ny):
    """The lane kernel (variant 0, with the list) against the node-by-node one (variant 3, without)."""
    pb = I.smooth_periodic(2, nx, ny, seed=3, amp=0.15)
    a, da = fields(pb, variant=0, learned_after=3)
    b, db = fields(pb, variant=3, learned_after=3)
    assert da["face_solves"] == db["face_solves"]
    for x, y in zip(a, b):
        assert rel_l1(x, y) <= 1e-5


@pytest.mark.parametrize("nx,ny", [(303, 127), (304, 127), (5, 3)])
def test_default_variant(nx, ny):
    """19 x 16 tiles and 20 x 16 (two tiles per SM on 152 SMs are 304), and a grid below a tile."""
    pb = I.smooth_periodic(2, nx, ny, seed=4, amp=0.1)
    a, da = fields(pb)
    for v in (0, 2):
        b, db = fields(pb, variant=v)
        assert da["face_solves"] == db["face_solves"]
        for x, y in zip(a, b):
            assert rel_l1(x, y) <= 1e-5
