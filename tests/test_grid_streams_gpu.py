"""A grid made while the default stream is busy and used on another stream: its
cleared arrays must not be cleared again behind the calls' backs."""
import numpy as np
import pytest
import torch

from paper_1908_11246_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


@pytest.mark.parametrize("n, even", [((130, 91), True), ((130, 91), False), ((20, 31, 72), True), ((300,), True)])
def test_new_grid_beside_a_busy_default_stream(n, even):
    from paper_1908_11246_gb300 import vup
    nd = len(n)
    rng = np.random.default_rng(sum(n))
    dens = I.random_densities(rng, 200, (-1.0,) * nd, (1.0,) * nd, sig=(0.4, 1.0), margin=0.2)
    y = sum(np.linspace(-1, 1, m).reshape([-1 if i == d else 1 for i in range(nd)]) ** 2 * (d + 1) if even else
            np.sin(np.linspace(0, 2, m) * (d + 1.3)).reshape([-1 if i == d else 1 for i in range(nd)])
            for d, m in enumerate(n))
    y = torch.as_tensor(np.array(np.broadcast_to(y, n), np.float64), device="cuda")
    dd = vup.densities_to_device(dens)
    prec = "fp64" if nd == 1 else "fp32"

    def one(stream):
        g = vup.Grid(n, (-1.0,) * nd, (1.0,) * nd)
        g.set_outputs(y, 30, stream=stream)
        return g, [t for t in g.propagate(dd, prec, central=False, stream=stream) if t is not None]

    g0, want = one(None)
    g0.sync()
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.empty(1 << 20, device="cuda")  # the side stream's memory exists before the default stream is busy
    torch.cuda._sleep(1 << 30)  # about half a second on the default stream
    with torch.cuda.stream(s):
        g, got = one(s)
    torch.cuda.synchronize()
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    for a, b in zip(want, [t for t in g.propagate(dd, prec, central=False) if t is not None]):
        assert torch.equal(a, b)
    g.sync()
    g.close()
    g0.close()
