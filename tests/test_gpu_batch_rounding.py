"""FP64 batches round as they always have.  A batch holds faces whose corrector cycles without converging, and
where it ends there depends on the last bits: in this one a pass that is the same in exact arithmetic moves the sums below by 5e-5.
The values are those of the node-by-node pass with the limiter's IEEE division, as first recorded; equal bits
give equal sums, and 1e-10 leaves room for the sums' own rounding."""
import numpy as np
import pytest

pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402

pytestmark = pytest.mark.gpu

RECORDED = [
    7.7671503180535666, -7.3521124581698558, -0.30830623908562771, 3.6031876316483467,
    -5.9481098009081315, -0.050893771480418293, -4.1641093183704116, -0.79993699521755479,
    -2.2310356869692702, 6.0900359035422866, -3.1091409026151653, 8.6459547323346744,
    3.5233040927469097, -0.69393624236869234, 3.0204001087884866, -1.0901956111880085,
    -0.28906344554646735, -0.68352359653073202, 5.0878466259835609, -1.1996404181571794,
    0.040869380529809152, -1.3469105166454578, 8.3915993348186095, 4.778026456124028,
]


def test_cycling_faces():
    rng = np.random.default_rng(5)
    n = 24
    lengths = rng.integers(100, 500, n)
    gammas = np.where(rng.integers(0, 2, n) == 0, 1.4, 5.0 / 3.0)
    rho, p = np.exp(rng.uniform(-1.15, 1.15, (n, 2))), np.exp(rng.uniform(-1.15, 1.15, (n, 2)))
    jump = rng.uniform(-0.5, 1.5, n) * np.sqrt(gammas * np.minimum(p[:, 0] / rho[:, 0], p[:, 1] / rho[:, 1]))
    side = np.concatenate([(2 * np.arange(k) + 1 > k).astype(int) for k in lengths])
    tube = np.repeat(np.arange(n), lengths)
    for variant in range(3):
        s = pond.BatchSolver(lengths, gammas, tau=1e-5, cfl=0.2, precision="fp64")
        s.set_variants(0, 0, variant)
        s.set_primitive(rho[tube, side], np.where(side == 0, 0.5, -0.5) * jump[tube], None, p[tube, side])
        s.step(40)
        d = s.sync(raise_on_error=False)
        assert d["nonconverged"] == 370
        E = np.asarray(s.moments(totals=False)[0][3])
        w = np.sin(np.arange(E.size) + 1.0)
        sums = np.add.reduceat(w * E, np.concatenate([[0], np.cumsum(lengths)[:-1]]))
        assert np.abs(sums - RECORDED).max() <= 1e-10
        s.close()
