"""The gradient kernel of the learned predictor at the edges of its work split: one row, one tile of
128 rows less, exactly and plus one, and more tiles than CTAs (so that some take two and the last
fewer); rows whose stride forbids 16-byte loads; and calls from more threads than there are
scratch slots."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2203_05477_gb300 as pond  # noqa: E402
from oracle import gauge_mlp as G  # noqa: E402

pytestmark = pytest.mark.gpu

BLOCKS = [(G.O_W1, G.O_B1), (G.O_B1, G.O_W2), (G.O_W2, G.O_B2), (G.O_B2, G.O_W3), (G.O_W3, G.O_B3), (G.O_B3, G.NPARAMS)]


def inputs(n, seed, width=52):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((n, width)).astype(np.float32)
    return G.init_params(seed).astype(np.float32), X


@pytest.mark.parametrize("n,width", [(1, 52), (127, 52), (128, 52), (129, 53), (300, 55), (304 * 128 + 77, 52)])
def test_gradient_at_the_edges(n, width):
    """The bounds of the other gradient tests: the loss to 1e-2, each tensor to 3e-2 of its scale
    (BF16 operands)."""
    p, X = inputs(n, n, width)
    d = torch.from_numpy(X).cuda()
    loss, g = pond.mlp_gradient(torch.from_numpy(p).cuda(), d, d)
    g = g.cpu().numpy()
    lref, gref = G.loss_and_grad(p.astype(np.float64), X[:, :48].astype(np.float64), X[:, 48:51].astype(np.float64), quantize=True)
    assert loss == pytest.approx(lref, rel=1e-2)
    for lo, hi in BLOCKS:
        scale = max(np.abs(gref[lo:hi]).max(), 1e-12)
        assert np.abs(g[lo:hi] - gref[lo:hi]).max() <= 3e-2 * scale, (lo, np.abs(g[lo:hi] - gref[lo:hi]).max() / scale)


def test_gradient_from_several_threads():
    """Six threads on their own streams: the same bits as one after the other."""
    jobs = []
    for k in range(6):
        p, X = inputs(500 + 997 * k, 40 + k)
        jobs.append((torch.from_numpy(p).cuda(), torch.from_numpy(X).cuda()))
    want = [pond.mlp_gradient(p, d, d) for p, d in jobs]
    torch.cuda.synchronize()
    got = [[] for _ in jobs]

    def work(k):
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(5):
                loss, g = pond.mlp_gradient(jobs[k][0], jobs[k][1], jobs[k][1])
                got[k].append((loss, g.clone()))
            torch.cuda.current_stream().synchronize()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for k, (loss, g) in enumerate(want):
        assert len(got[k]) == 5
        for l2, g2 in got[k]:
            assert l2 == loss and torch.equal(g2, g)
