"""Steps captured into a graph of the caller's: an odd number of them, replayed several times and between other
steps, on every kind of finite-volume grid, gives the bits of the same steps run in place without a graph.  (The
fused step changes buffers, so a graph of an odd number of fused steps would start from the same
buffer each time.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from paper_2203_05477_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

CASES = {
    "tube_short": (lambda: I.sod_400(), 0),
    "tube": (lambda: I.smooth_periodic(1, 20000, 1, seed=1, amp=0.15), 0),
    "grid": (lambda: I.smooth_periodic(2, 45, 37, seed=1, amp=0.15), 0),
    "grid_fused": (lambda: I.smooth_periodic(2, 45, 37, seed=1, amp=0.15), 1),
}


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("before", [0, 1, 33])
@pytest.mark.parametrize("name", sorted(CASES))
def test_replayed_steps(name, before, precision):
    make, fused = CASES[name]
    pb = make()
    out = []
    for captured in (True, False):
        stream = torch.cuda.Stream()
        s = pond.Solver(pb, precision=precision, tau=1e-5, cfl=0.2, stream=stream)
        if fused:
            s.set_variants(0, 0, fused)
        s.set_primitive()
        s.step(before)   # the default step, or the fused one: the buffers as they come
        if captured:
            s.sync()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=stream):
                s.step(3)
            with torch.cuda.stream(stream):
                g.replay()
                g.replay()
                s.step(1)
                g.replay()
                s.step(40)
                g.replay()
        else:
            s.set_variants(0, 0, 0)
            s.step(3 + 3 + 1 + 3 + 40 + 3)
        d = s.sync()
        assert d["steps"] == before + 53 and d["nonphysical"] == 0
        out.append([*s.state(), *[a for a in s.face_gauges() if a is not None]])
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
