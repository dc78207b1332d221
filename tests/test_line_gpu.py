"""1-D grids in FP64 at the sizes where the cluster of CTAs per density changes
(one density, a few, many; axes shorter than a CTA, ragged, the longest; up to
the most bins), every density kind, means outside the domain, against the FP64
oracle at the 1-D path's tolerance (1e-12 of the condition scale)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1908_11246_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


@pytest.mark.parametrize("n, K, B", [(7, 3, 5), (100, 1, 300), (1023, 40, 64), (4097, 700, 64), (6145, 9, 2048),
                                     (32767, 2, 8192), (300, 3000, 1)])
def test_line_matches_oracle(n, K, B):
    from paper_1908_11246_gb300 import vup
    rng = np.random.default_rng(n + K)
    dens = I.random_densities(rng, K, (-5.0,), (5.0,), kinds=(I.GAUSS, I.UNIFORM, I.TRUNCNORM),
                              sig=(max(0.03, 15.0 / n), max(1.0, 22.0 / n)),
                              width=(max(0.2, 30.0 / n), 6.0))
    far = np.arange(K) % 7 == 3  # means past the domain's ends: only a tail is left
    dens.kind[far] = I.GAUSS
    dens.mu[far] = 5.0 + 3.0 * rng.random((int(far.sum()), 1))
    dens.sigma[far] = np.maximum(dens.sigma[far], 0.2)
    prob = I.Problem("line", (n,), (-5.0,), (5.0,), I.MODEL_SIN_QUAD_1D, (1.0, 0.1), dens, B, 4, "fp64")
    ref = O.solve(prob, rows=np.arange(K))
    one = np.zeros(n, np.int32)
    scale = O.propagate(prob.n, prob.lo, prob.hi, np.abs(ref["y"]), one, 1, 4, dens, rows=np.arange(K))["raw"]
    g = vup.Grid(prob.n, prob.lo, prob.hi)
    g.eval_model(prob.model_id, prob.theta, B)
    dd = vup.densities_to_device(dens)
    raw, cen, hist = g.propagate(dd, "fp64")
    hist_only = g.propagate(dd, "fp64", moments=False, central=False)[2]
    g.sync()
    raw, cen = raw.cpu().numpy(), cen.cpu().numpy()
    assert (np.abs(raw - ref["raw"]) <= 1e-12 * scale).all()
    assert (np.abs(cen - ref["central"]) <= 1e-12 * 39 * scale).all()
    assert np.abs(hist.cpu().numpy() - ref["hist"]).max() <= 1e-6
    assert (hist_only == hist).all()
    g.close()
