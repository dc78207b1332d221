"""vup_hist_walk tells what the histograms walk (sizes, layout, stream and counts
of the merged grid) and vup_grid_info keeps describing the grid itself, both
against counts from the device's bins on the host, the stream against the
layout build's cost rule."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1908_11246_gb300 import inputs as I
from tests.test_hist_fold_gpu import NAMES, _case
from tests.test_hist_streams_gpu import layout_counts

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def merged(b):
    """The bins with equal slices of every axis merged where at most 5/8 remain."""
    keep = []
    for d in range(b.ndim):
        first = {}
        for i in range(b.shape[d]):
            first.setdefault(np.take(b, i, axis=d).tobytes(), i)
        heads = sorted(first.values())
        keep.append(heads if 8 * len(heads) <= 5 * b.shape[d] else range(b.shape[d]))
    return b[np.ix_(*keep)]


def cheaper_stream(N, ndim, runs, ivs, recs):
    rec = (16 + 6 * (ndim - 1)) * recs + 6 * (ivs + 2 * recs)
    if rec < 4 * N and rec <= 19 * ivs:
        return 2
    return 1 if 19 * ivs < 4 * N + 20 * runs else 0


@pytest.mark.parametrize("name", NAMES)
def test_walk_is_that_of_the_merged_grid(name):
    from paper_1908_11246_gb300 import vup
    n, y, B = _case(name)
    y = np.ascontiguousarray(y, dtype=np.float64)
    b = O.bins(y.ravel(), B)[0].reshape(n)
    m = merged(b)
    g = vup.Grid(n, (-1.0,) * len(n), (2.0,) * len(n))
    with pytest.raises(vup.VUPError) as e:
        g.hist_walk()
    assert e.value.status == vup.VUP_ERR_STATE
    y = torch.as_tensor(y, device="cuda")
    g.set_outputs(y, B)
    for kind in (-1, 0, 1, 2, -1):
        g.set_hist_stream(kind)
        w = g.hist_walk()
        assert tuple(w.n[:len(n)]) == m.shape and w.N == m.size
        counts = [layout_counts(m, B, l) for l in range(2 if len(n) == 2 else 1)]
        assert w.layout == (1 if len(counts) == 2 and counts[1][1] < counts[0][1] else 0)
        runs, ivs, recs = counts[w.layout]
        assert w.stream == (cheaper_stream(m.size, len(n), runs, ivs, recs) if kind < 0 else kind)
        assert (w.intervals, w.records) == (ivs, recs)
        assert w.runs == (0 if w.stream == 2 else runs)
        info = g.info()
        runs, ivs, recs = layout_counts(b, B, info.hist_layout)
        assert (info.hist_intervals, info.hist_records) == (ivs, recs)
        assert info.hist_runs == runs or (info.hist_stream == 2 and info.hist_runs == 0)
        # a second look builds nothing, and finds the same
        vup.vup_profile(True)
        again, wagain = g.info(), g.hist_walk()
        vup.vup_profile(False)
        assert not vup.vup_profile_read()
        assert bytes(again) == bytes(info) and bytes(wagain) == bytes(w)
    # another model: counts anew
    g.set_outputs(torch.flip(y, (0,)).contiguous(), B)
    flipped = np.ascontiguousarray(b[::-1])
    info = g.info()
    assert layout_counts(flipped, B, info.hist_layout)[1:] == (info.hist_intervals, info.hist_records)
    g.close()


@pytest.mark.parametrize("name", ["c2", "c3"])
def test_walk_of_full_size_workloads(name):
    """The counts and the choice at full size, where the merged grid's stream may be
    another than the grid's own (three axes: intervals where the grid has points)."""
    from paper_1908_11246_gb300 import vup
    p = I.config(name)
    g = vup.Grid(p.n, p.lo, p.hi)
    g.eval_model(p.model_id, p.theta, p.n_bins, p.n_moments)
    w = g.hist_walk()
    m = merged(g.array("bins").cpu().numpy().reshape(p.n))
    assert tuple(w.n[:len(p.n)]) == m.shape
    runs, ivs, recs = layout_counts(m, p.n_bins, w.layout)
    assert w.stream == cheaper_stream(m.size, len(p.n), runs, ivs, recs)
    assert (w.intervals, w.records) == (ivs, recs)
    g.close()


def test_walk_argument_errors():
    from paper_1908_11246_gb300 import vup
    g = vup.Grid((16,), (0.0,), (1.0,))
    g.set_outputs(torch.zeros(16, dtype=torch.float64, device="cuda"), 4)
    with pytest.raises(vup.VUPError) as e:
        g.hist_walk()
    assert e.value.status == vup.VUP_ERR_INVALID_ARG
    g.close()
