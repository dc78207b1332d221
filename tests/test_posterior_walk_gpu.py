"""Posterior means in one walk, at the sizes where it changes: one and more than
one tile of 64 densities, parts of a long axis, equal slices merged or not,
three axes with the rest factors staged or not, bins without points, H wanted or
not.  Each against the oracle's plain definition on bins that hold mass (2e-5 of
the axis' extent, the tolerance of the posterior tests) and H at 1e-6."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1908_11246_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


@pytest.mark.parametrize("n, K, B, even", [((40, 33), 1, 12, True), ((40, 33), 65, 300, False), ((900, 50), 130, 40, False),
                                           ((50, 901), 70, 40, True), ((20, 24, 30), 66, 25, True),
                                           ((9, 520, 16), 40, 30, False), ((3, 4100, 5), 5, 9, True)])
def test_one_walk_matches_definition(n, K, B, even):
    from paper_1908_11246_gb300 import vup
    nd = len(n)
    lo, hi = (-1.0,) * nd, (1.0,) * nd
    rng = np.random.default_rng(sum(n))
    dens = I.random_densities(rng, K, lo, hi, sig=(0.5, 1.0), margin=0.2)
    x = [lo[d] + (np.arange(n[d]) + 0.5) * ((hi[d] - lo[d]) / n[d]) for d in range(nd)]
    y = 0.0
    for d in range(nd):
        s = [1] * nd
        s[d] = -1
        y = y + ((d + 1.0) * x[d] ** 2 if even else np.sin((d + 1.3) * x[d]) + 0.2 * x[d]).reshape(s)
    y = np.array(np.broadcast_to(y, n), dtype=np.float64)
    b, _, _ = O.bins(y.ravel(), B)
    g = vup.Grid(n, lo, hi)
    g.set_outputs(torch.as_tensor(y, device="cuda"), B)
    dd = vup.densities_to_device(dens)
    hist = torch.empty((K, B), dtype=torch.float32, device="cuda")
    post = torch.empty((K, B, nd), dtype=torch.float32, device="cuda")
    again = torch.empty_like(post)
    vup.vup_posterior_means(g.h, vup.make_densities(dd), hist, post)
    vup.vup_posterior_means(g.h, vup.make_densities(dd), None, again)
    g.sync()
    assert torch.equal(post, again)
    # the plain definition in FP64
    w = [np.exp(-0.5 * ((x[d][None, :] - dens.mu[:, d:d + 1]) / dens.sigma[:, d:d + 1]) ** 2) for d in range(nd)]
    w = [v / v.sum(1, keepdims=True) for v in w]
    hist, post = hist.cpu().numpy(), post.cpu().numpy()
    grids = np.meshgrid(*x, indexing="ij")
    for k in range(0, K, max(1, K // 8)):
        W = w[0][k]
        for d in range(1, nd):
            W = np.multiply.outer(W, w[d][k])
        W = W.ravel()
        H = np.bincount(b, W, B)
        assert np.abs(hist[k] - H).max() <= 1e-6
        for d in range(nd):
            m = np.bincount(b, W * grids[d].ravel(), B)
            ok = H > 1e-12
            assert np.abs(post[k, ok, d] - m[ok] / H[ok]).max() <= 2e-5 * 2.0
            assert (post[k, H == 0, d] == 0).all()
    g.close()
