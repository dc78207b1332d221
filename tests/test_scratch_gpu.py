"""Device memory that calls take on top of the grid's and the densities' own
scratch, against the sizes the documentation gives (2 MB of the allocator's
granularity per buffer)."""
import numpy as np
import pytest
import torch

from paper_1908_11246_gb300 import inputs as I

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def _cap(n):
    return (5 * n + 7) // 8


def _setup(n, K, B):
    from paper_1908_11246_gb300 import vup
    nd = len(n)
    dens = I.random_densities(np.random.default_rng(5), K, (-1.0,) * nd, (1.0,) * nd, sig=(0.4, 1.0), margin=0.2)
    y = 0.0
    for d in range(nd):
        y = y + torch.linspace(-1, 1, n[d], dtype=torch.float64, device="cuda").square().reshape(
            [-1 if q == d else 1 for q in range(nd)]) * (d + 1)
    g = vup.Grid(n, (-1.0,) * nd, (1.0,) * nd)
    g.set_outputs(y.expand(n).contiguous(), B)
    return g, vup.densities_to_device(dens), B


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


@pytest.mark.parametrize("n, K", [((1024, 1024), 16384), ((300, 2000), 16384), ((96, 96, 900), 16384)])
def test_merged_tables_are_those_of_the_rest_axes(n, K):
    """2-D: the larger of the two axes' (one is gathered); 3-D: the first two's."""
    from paper_1908_11246_gb300 import vup
    g, dd, B = _setup(n, K, 16)
    d = vup.make_densities(dd)
    raw = torch.empty((K, 4), dtype=torch.float64, device="cuda")
    hist = torch.empty((K, B), dtype=torch.float32, device="cuda")
    g.info()  # the layout is there
    vup.vup_propagate(g.h, d, vup.VUP_FP32, raw, None, None)
    before = _used()
    vup.vup_propagate(g.h, d, vup.VUP_FP32, raw, None, hist)
    rows = max(_cap(n[0]), _cap(n[1])) if len(n) == 2 else _cap(n[0]) + _cap(n[1])
    assert _used() - before <= 4 * rows * K + 6 * MB
    before = _used()
    vup.vup_propagate(g.h, d, vup.VUP_FP32, raw, None, hist)
    assert _used() == before
    g.sync()
    g.close()


@pytest.mark.parametrize("n, K, B", [((300, 2000), 3000, 5000), ((20, 24, 900), 2500, 8192)])
def test_posterior_sums_are_held_for_blocks_of_densities(n, K, B):
    """Many keys (6 and 3 parts x B bins): the walk's sums stay within 512 MB beside the
    weighted factors, and the blocks' seams give what calls of a few densities give."""
    from paper_1908_11246_gb300 import vup
    nd = len(n)
    g, dd, B = _setup(n, K, B)
    K_pad = -(-K // 128) * 128
    hist = torch.empty((K, B), dtype=torch.float32, device="cuda")
    post = torch.empty((K, B, nd), dtype=torch.float32, device="cuda")
    g.propagate(dd, "fp32", moments=False, central=False)  # the scratch of a propagation
    torch.cuda.empty_cache()
    before = _used()
    vup.vup_posterior_means(g.h, vup.make_densities(dd), hist, post)
    assert _used() - before <= 4 * sum(n) * K_pad + 512 * MB + 6 * MB
    for k0 in [*range(0, K - 200, 97), K - 200]:
        part = {q: v[k0:k0 + 200].contiguous() for q, v in dd.items()}
        h, p = torch.empty_like(hist[:200]), torch.empty_like(post[:200])
        vup.vup_posterior_means(g.h, vup.make_densities(part), h, p)
        torch.cuda.synchronize()
        # the same sums in the same order, whatever the block
        assert torch.equal(h, hist[k0:k0 + 200]) and torch.equal(p, post[k0:k0 + 200])
    g.sync()
    g.close()
