"""FP64 moments and sensitivities of 1-D grids whose sums lie far out in the
densities' tails: outputs so steep that E[y^4] sits near 16 sigma, outputs that
are zero but beyond 20 and 30 sigma (tail probabilities down to 1e-167), means
outside the domain, against the FP64 oracle; and outputs that are not finite.

Tolerance: the path's 1e-12 of the condition scale.  A weight's relative error
is |u| du with du <= 2^-51 |x|max / sigma, below 5e-13 for the cases here."""
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


def _gauss(mu, sigma):
    K = len(mu)
    col = lambda v: np.asarray(v, np.float64).reshape(K, 1)
    return I.Densities(np.full((K, 1), I.GAUSS, np.uint8), col(mu), col(sigma), np.zeros((K, 1)), np.zeros((K, 1)))


def _grid(n, lo, hi, y, B):
    from paper_1908_11246_gb300 import vup
    g = vup.Grid((n,), (lo,), (hi,))
    g.set_outputs(torch.as_tensor(y, device="cuda"), B)
    return g


def _case(name):
    """(n, lo, hi, mu, sigma, y)"""
    if name == "steep":
        n, lo, hi, mu, sigma = 4096, -1.0, 1.0, (0.0, -0.15, -0.05), (0.05, 0.045, 0.05)
        rate = 80.0
    elif name == "steep_ragged":
        n, lo, hi, mu, sigma = 3001, -5.0, 5.0, (0.1, -0.4, -5.2), (0.3, 0.28, 0.4)
        rate = 13.0
    else:
        n, lo, hi, mu, sigma = 2500, 0.0, 1.0, (0.02, 0.1, 0.3), (0.03, 0.02, 0.015)
        rate = 0.0
    x = lo + (np.arange(n) + 0.5) * ((hi - lo) / n)
    y = 1e-8 * np.exp(rate * x) if rate else np.where(x > 0.65, 0.5, 0.0)
    return n, lo, hi, _gauss(mu, sigma), y


@pytest.mark.parametrize("name", ["steep", "steep_ragged", "tail_only"])
def test_tail_sums_match_oracle(name):
    from paper_1908_11246_gb300 import vup
    n, lo, hi, dens, y = _case(name)
    B, J = 40, 4
    b, _, _ = O.bins(y, B)
    args = ((n,), (lo,), (hi,))
    ref = O.propagate(*args, y, b, B, J, dens)
    scale = O.propagate(*args, np.abs(y), np.zeros(n, np.int32), 1, J, dens)["raw"]
    dmu, dsg = O.ipsa(*args, y, J, dens)
    cmu, csg = O.ipsa_scale(*args, y, J, dens)
    g = _grid(n, lo, hi, y, B)
    dd = vup.densities_to_device(dens)
    raw, cen, hist = (t.cpu().numpy() for t in g.propagate(dd, "fp64"))
    gmu, gsg = (t.cpu().numpy().astype(np.float64) for t in g.ipsa(dd, "fp64"))
    g.sync()
    assert (np.abs(raw - ref["raw"]) <= 1e-12 * scale).all()
    assert (np.abs(cen - ref["central"]) <= 1e-12 * 39 * scale).all()
    assert np.abs(hist - ref["hist"]).max() <= 1e-6
    for got, want, cond in ((gmu, dmu, cmu), (gsg, dsg, csg)):  # FP32 outputs, the smallest of them subnormal
        assert (np.abs(got - want) <= 1e-12 * cond + 2.0 ** -23 * np.abs(want) + 1e-44).all()
    g.close()


def test_output_that_is_not_finite_reaches_every_density():
    from paper_1908_11246_gb300 import vup
    n = 1000
    y = np.linspace(0.0, 1.0, n)
    y[-1] = np.inf
    dens = _gauss((0.1, 0.2), (0.004, 0.01))
    g = _grid(n, 0.0, 1.0, y, 16)
    raw = g.propagate(vup.densities_to_device(dens), "fp64", central=False, hist=False)[0]
    assert not np.isfinite(raw.cpu().numpy()).any()  # 0 times infinity
    g.close()
