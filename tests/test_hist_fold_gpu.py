"""Equal slices of the bin grid are merged before the histogram walks (two
indices of an axis whose points all fall in the same bins): outputs with
repeated, mirrored, ignored and almost-equal slices against the FP64 oracle,
each stream forced, and the counts of vup_grid_info, which describe the grid
itself.  Tolerance: the histogram gate (1e-6 absolute per bin)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1908_11246_gb300 import inputs as I
from tests.test_hist_streams_gpu import layout_counts

pytestmark = pytest.mark.gpu

HIST_TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def _case(name):
    """(sizes, outputs y on the grid, bins)"""
    rng = np.random.default_rng(71)
    if name == "mirror_odd":           # one unpaired slice per axis
        a, b = np.linspace(-1, 1, 129), np.linspace(-1, 1, 77)
        return (129, 77), np.add.outer(a * a, 3 * np.abs(b)), 50
    if name == "ignored_axis":         # one class of every slice
        return (60, 500), np.tile(np.sin(np.linspace(0, 3, 60))[:, None], (1, 500)), 33
    if name == "repeats":              # members scattered over the axis, parts of several tiles
        base = np.cumsum(rng.uniform(0.1, 1, (300, 90)), 0)
        return (900, 90), base[rng.integers(0, 300, 900)], 64
    if name == "one_point_off":        # mirrored but for single points: those slices stay apart
        a = np.linspace(-1, 1, 200)
        y = np.add.outer(a * a, np.linspace(0, 1, 64))
        y[150:190, 7] += 0.2
        return (200, 64), y, 40
    if name == "few_equal":            # more than 5/8 distinct: nothing is merged
        base = rng.uniform(0, 1, (100, 80))
        return (100, 80), base[np.minimum(np.arange(100), 65)], 21
    if name == "volume":               # every axis mirrored, one odd
        a, b, c = np.linspace(-1, 1, 20), np.linspace(-1, 1, 31), np.linspace(-2, 2, 72)
        return (20, 31, 72), (a * a)[:, None, None] + np.abs(b)[None, :, None] * (c ** 4)[None, None, :], 100
    return (1, 40), np.linspace(0, 1, 40)[None, :] ** 2, 8   # an axis of one index


NAMES = ["mirror_odd", "ignored_axis", "repeats", "one_point_off", "few_equal", "volume", "single"]


@pytest.mark.parametrize("name", NAMES)
def test_merged_slices_match_oracle(name):
    from paper_1908_11246_gb300 import vup
    n, y, B = _case(name)
    nd = len(n)
    lo, hi = (-1.0,) * nd, (2.0,) * nd
    K = 150
    dens = I.random_densities(np.random.default_rng(72), K, lo, hi, kinds=(I.GAUSS, I.UNIFORM) if min(n) > 16 else
                              (I.GAUSS,), sig=(0.2, 1.0), width=(0.6, 2.0), margin=0.1)
    y = np.ascontiguousarray(y, dtype=np.float64)
    b, _, _ = O.bins(y.ravel(), B)
    ref = O.propagate(n, lo, hi, y.ravel(), b, B, 4, dens, rows=np.arange(K))["hist"]
    g = vup.Grid(n, lo, hi)
    g.set_outputs(torch.as_tensor(y, device="cuda"), B)
    dd = vup.densities_to_device(dens)
    for kind in (-1, 0, 1, 2):
        g.set_hist_stream(kind)
        for _ in range(2):  # the second call keeps the layout
            _, _, hs = g.propagate(dd, "fp32")
            g.sync()
            assert np.abs(hs.cpu().numpy() - ref).max() <= HIST_TOL, (name, kind)
        info = g.info()
        runs, ivs, recs = layout_counts(b.reshape(n), B, info.hist_layout)
        assert (info.hist_intervals, info.hist_records) == (ivs, recs)
        assert info.hist_runs == runs or (info.hist_stream == 2 and info.hist_runs == 0)
    g.close()


def test_merged_slices_batched():
    """An even model (every axis folded) beside one that is not, in one batch."""
    from paper_1908_11246_gb300 import vup
    probs = []
    for i, theta in enumerate(((0.0, 0.0, 1.0, 0.0, 2.0), (0.0, 1.0, 0.5, 0.3, 0.2))):
        lo, hi = (-1.0, -2.0), (1.0, 2.0)
        dens = I.random_densities(np.random.default_rng(80 + i), 300, lo, hi, sig=(0.1, 0.8))
        probs.append(I.Problem(f"poly{i}", (130, 91), lo, hi, I.MODEL_POLY, theta, dens, 60))
    grids, dds = [], []
    for p in probs:
        g = vup.Grid(p.n, p.lo, p.hi)
        g.eval_model(p.model_id, p.theta, p.n_bins)
        grids.append(g)
        dds.append(vup.densities_to_device(p.dens))
    out = vup.propagate_batched(grids, dds, "fp32")
    vup.propagate_batched(grids, dds, "fp32", out=out)
    for p, g, hs in zip(probs, grids, out[1]):
        g.sync()
        ref = O.solve(p, rows=np.arange(p.K))["hist"]
        assert np.abs(hs.cpu().numpy() - ref).max() <= HIST_TOL


# records per part from fewer than one chunk per warp to several rounds of chunks for every warp
@pytest.mark.parametrize("n0,n1,B", [(24, 40, 8), (200, 300, 30), (401, 500, 60), (640, 900, 64), (1800, 1100, 500)])
def test_record_chunks_match_oracle(n0, n1, B):
    from paper_1908_11246_gb300 import vup
    lo, hi = (-1.0, -1.0), (2.0, 2.0)
    y = np.add.outer(np.linspace(-1, 1, n0) ** 2, 3 * np.abs(np.linspace(-1, 1, n1)))
    K = 130
    dens = I.random_densities(np.random.default_rng(90), K, lo, hi, kinds=(I.GAUSS,), sig=(0.2, 1.0), margin=0.1)
    b, _, _ = O.bins(y.ravel(), B)
    ref = O.propagate((n0, n1), lo, hi, y.ravel(), b, B, 4, dens, rows=np.arange(K))["hist"]
    g = vup.Grid((n0, n1), lo, hi)
    g.set_outputs(torch.as_tensor(y, device="cuda"), B)
    g.set_hist_stream(2)
    _, _, hs = g.propagate(vup.densities_to_device(dens), "fp32")
    g.sync()
    assert np.abs(hs.cpu().numpy() - ref).max() <= HIST_TOL
    g.close()
