"""The FP64 van Leer quotient ab / (a + b) of the face kernels (a hardware seed and two Newton steps) against the
division, over magnitudes from 1e-140 to 1e140, ratios up to 1e6 either way and all signs.

It is within 2^-57, a sixteenth of a unit in the last place, of the quotient before its one rounding: never more
than one unit off, and rounded to another neighbour than the division in at most one of eight draws."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2203_05477_gb300 import _build  # noqa: E402

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pond_vec.cuh"
__global__ void quotients(const double *a, const double *b, double *q, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) q[i] = pond::vanleer_half(a[i], b[i]);
}
extern "C" int run(const double *a, const double *b, double *q, int n)
{
    quotients<<<(n + 255) / 256, 256>>>(a, b, q, n);
    return int(cudaDeviceSynchronize());
}
"""


def test_quotient(tmp_path):
    src, lib = tmp_path / "quotient.cu", tmp_path / "quotient.so"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", *_build.FLAGS, "-I", _build.CSRC, "-shared", "-o", str(lib), str(src)], check=True)
    rng = np.random.default_rng(0)
    n = 1 << 20
    a = 10.0 ** rng.uniform(-140, 140, n) * rng.choice([-1.0, 1.0], n)
    b = a * 10.0 ** rng.uniform(-6, 6, n) * rng.choice([1.0, 1.0, 1.0, -1.0], n)
    a[:6], b[:6] = [0.0, 1.0, -0.0, np.nan, 1.0, 3.0], [0.0, 0.0, 1.0, 1.0, -1.0, 3.0]
    da, db = (torch.from_numpy(x).cuda() for x in (a, b))
    dq = torch.empty_like(da)
    assert ctypes.CDLL(str(lib)).run(*[ctypes.c_void_p(t.data_ptr()) for t in (da, db, dq)], n) == 0
    q = dq.cpu().numpy()
    with np.errstate(invalid="ignore", divide="ignore"):
        ab = a * b
        want = np.where(ab > 0.0, ab / (a + b), 0.0)
    off = np.abs(q - want) / np.spacing(np.abs(want))
    assert not np.isnan(q).any() and (q[~(ab > 0.0)] == 0.0).all()
    assert off.max() <= 1.0
    assert np.mean(off > 0.0) <= 0.125
