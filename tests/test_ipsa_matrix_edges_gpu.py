"""IPSA matrix columns whose estimated value is not finite: NaN puts a column's
mass in no deviation bin, an infinity in the first or last; the other columns
are the oracle's bit for bit.  And outputs whose size dwarfs their range, where
the FP64 expression of a deviation bin is itself rounded by part of a bin."""
import numpy as np
import pytest
import torch

from oracle import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def _grid(y, B):
    from paper_1908_11246_gb300 import vup
    g = vup.Grid(y.shape, (0.0,) * y.ndim, (1.0,) * y.ndim)
    g.set_outputs(torch.as_tensor(y, device="cuda"), B)
    return g


@pytest.mark.parametrize("B, nd", [(1, 1), (100, 37), (300, 701), (8192, 8192)])
def test_values_that_are_not_finite(B, nd):
    from paper_1908_11246_gb300 import vup
    rng = np.random.default_rng(B + nd)
    g = _grid(np.linspace(-1.0, 2.0, 3000).reshape(60, 50), B)
    hist = rng.random((40, B)).astype(np.float32)
    yref = rng.uniform(-1.0, 2.0, 40)
    yref[3::9], yref[4::9], yref[5::9] = np.nan, np.inf, -np.inf
    out = torch.full((40, nd), -1.0, dtype=torch.float32, device="cuda")
    vup.vup_ipsa_matrix(g.h, torch.as_tensor(hist, device="cuda"), torch.as_tensor(yref, device="cuda"), nd, -3.0,
                        3.0, out)
    g.sync()
    ok = np.isfinite(yref)
    want = np.zeros((40, nd), np.float32)
    want[ok] = O.ipsa_matrix(hist[ok].astype(np.float64), -1.0, 2.0, yref[ok], nd, -3.0, 3.0).astype(np.float32)
    total = np.cumsum(hist.astype(np.float64), axis=1)[:, -1].astype(np.float32)  # in increasing b
    want[yref == np.inf, 0] = total[yref == np.inf]
    want[yref == -np.inf, nd - 1] = total[yref == -np.inf]
    np.testing.assert_array_equal(out.cpu().numpy(), want)
    g.close()


def test_outputs_that_are_not_finite():
    """A range with an infinite end gives no deviation bin to any column."""
    from paper_1908_11246_gb300 import vup
    y = np.linspace(-1.0, 2.0, 3000).reshape(60, 50)
    y[0, 0] = -np.inf
    g = _grid(y, 64)
    out = torch.full((5, 20), -1.0, dtype=torch.float32, device="cuda")
    vup.vup_ipsa_matrix(g.h, torch.ones((5, 64), device="cuda"), torch.zeros(5, dtype=torch.float64, device="cuda"),
                        20, -1.0, 1.0, out)
    g.sync()
    assert (out == 0).all()
    g.close()


@pytest.mark.parametrize("offset", [0.0, 1e6, -1e9, 3e9, 1e12, -1e15])
@pytest.mark.parametrize("B, nd", [(1000, 1000), (333, 2048), (4096, 700)])
def test_offset_outputs_match_oracle(offset, B, nd):
    from paper_1908_11246_gb300 import vup
    rng = np.random.default_rng(B + nd)
    y = np.linspace(-1.0, 2.0, 3000).reshape(60, 50) + offset
    g = _grid(y, B)
    info = g.info()
    hist = rng.random((60, B)).astype(np.float32)
    yref = offset + rng.uniform(-1.0, 2.0, 60)
    for dlo, dhi in ((-3.0, 3.0), (-0.7, 4.1)):
        out = torch.empty((60, nd), dtype=torch.float32, device="cuda")
        vup.vup_ipsa_matrix(g.h, torch.as_tensor(hist, device="cuda"), torch.as_tensor(yref, device="cuda"), nd, dlo,
                            dhi, out)
        g.sync()
        want = O.ipsa_matrix(hist.astype(np.float64), info.ymin, info.ymax, yref, nd, dlo, dhi)
        np.testing.assert_array_equal(out.cpu().numpy(), want.astype(np.float32))
    g.close()
