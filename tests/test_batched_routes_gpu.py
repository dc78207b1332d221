"""Batches whose instances want different outputs, against the FP64 oracle: an
instance without a histogram may have no layout yet, or merged tables from an
earlier call with fewer densities."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1908_11246_gb300 import inputs as I
from tests import helpers as Hp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def _poly(i, n, K, even):
    lo, hi = (-1.0, -2.0), (1.0, 2.0)
    theta = (0.0, 0.0, 1.0, 0.0, 2.0) if even else (0.0, 1.0, 0.5, 0.3, 0.2)
    dens = I.random_densities(np.random.default_rng(600 + i), K, lo, hi, sig=(0.1, 0.8))
    return I.Problem(f"poly{i}", n, lo, hi, I.MODEL_POLY, theta, dens, 60)


def _check(p, raw, hist, precision):
    rows = np.arange(p.K)
    res = O.solve(p, rows=rows, threads=Hp.oracle_threads())
    if raw is not None:
        scale = Hp.abs_moment_scale(p, res["y"], rows)
        Hp.check_moments(raw.cpu().numpy(), res["raw"], scale, Hp.TOL[precision], what=p.name)
    if hist is not None:
        amb = Hp.ambiguous_points(res["y"], res["bins"], p.n_bins)
        Hp.check_hist(hist.cpu().numpy(), res["hist"], Hp.ambiguous_mass(p, amb, rows))


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_instances_without_histogram(precision):
    """0: merged tables from a call with fewer densities; 1: no layout, on memory
    of closed grids; 2, 3: histograms with and without merged slices; 4: nothing wanted."""
    from paper_1908_11246_gb300 import vup
    for n in ((64, 90), (130, 91)):  # closed grids leave their merged sizes behind in freed memory
        p = _poly(9, n, 200, True)
        g = vup.Grid(p.n, p.lo, p.hi)
        g.eval_model(p.model_id, p.theta, p.n_bins)
        g.propagate(vup.densities_to_device(p.dens), precision)
        g.sync()
        g.close()
    probs = [_poly(0, (130, 91), 3000, True), _poly(1, (64, 90), 700, True), _poly(2, (120, 80), 500, True),
             _poly(3, (77, 130), 300, False), _poly(4, (40, 50), 260, True)]
    grids, dds = [], []
    for p in probs:
        g = vup.Grid(p.n, p.lo, p.hi)
        g.eval_model(p.model_id, p.theta, p.n_bins)
        grids.append(g)
        dds.append(vup.densities_to_device(p.dens))
    few = _poly(7, (130, 91), 100, True)
    _check(few, *grids[0].propagate(vup.densities_to_device(few.dens), precision, central=False)[::2], precision)
    raws, hists = vup.batched_outputs(grids, dds)
    hists[0] = hists[1] = hists[4] = raws[4] = raws[3] = None
    for _ in range(2):  # the second call replays the graph
        for t in raws + hists:
            if t is not None:
                t.fill_(-1)
        vup.propagate_batched(grids, dds, precision, out=(raws, hists))
        for g in grids:
            g.sync()
        for p, r, h in zip(probs, raws, hists):
            _check(p, r, h, precision)
    # and the instances without a histogram in a call of their own
    for p, g, dd in zip(probs, grids, dds):
        r, _, h = g.propagate(dd, precision, central=False)
        g.sync()
        _check(p, r, h, precision)
        g.close()


def _oscillators():
    return I.oscillator_batch(23, n_inst=8, side=(24, 400), kk=(40, 900), n_bins=128) + [_poly(5, (90, 61), 300, True)]


def _grids(probs):
    from paper_1908_11246_gb300 import vup
    out = []
    for p in probs:
        g = vup.Grid(p.n, p.lo, p.hi)
        g.eval_model(p.model_id, p.theta, p.n_bins, p.n_moments)
        out.append(g)
    return out


def test_histograms_do_not_depend_on_which_call_came_first():
    """One instance alone, in a batch, in a batch first and then alone, and alone
    after vup_grid_info has looked at the counts: the same bits, on grids of each
    order's own (the documented identity of the batched and the one-instance path)."""
    from paper_1908_11246_gb300 import vup
    probs = _oscillators()
    dds = [vup.densities_to_device(p.dens) for p in probs]

    def alone(grids):
        return [g.propagate(dd, "fp32", moments=False, central=False)[2] for g, dd in zip(grids, dds)]

    def batch(grids):
        return vup.propagate_batched(grids, dds, "fp32", moments=False)[1]

    def looked_at(grids):
        for g in grids:
            g.info()
        return alone(grids)

    first, second, third, fourth = (_grids(probs) for _ in range(4))
    results = dict(alone=alone(first), batch_after_alone=batch(first), batch=batch(second), alone_after_batch=alone(second),
                   looked_at=looked_at(third), batch_after_look=batch(third))
    batch(fourth)
    results["batch_then_look_then_alone"] = looked_at(fourth)
    import torch
    torch.cuda.synchronize()
    for name, hs in results.items():
        for p, a, b in zip(probs, results["alone"], hs):
            np.testing.assert_array_equal(b.cpu().numpy(), a.cpu().numpy(), err_msg=f"{name} {p.name}")


@pytest.mark.parametrize("precision", ["fp32", "bf16x3"])
def test_new_grids_never_replay_the_graph_of_destroyed_ones(precision):
    """Batches of new grids on the same densities and output buffers, the ones before
    destroyed: sizes, buffers and (as the allocators go) addresses repeat."""
    from paper_1908_11246_gb300 import vup
    probs = I.oscillator_batch(29, n_inst=4, side=(32, 191), kk=(64, 1500), n_bins=67)
    dds = [vup.densities_to_device(p.dens) for p in probs]
    grids = _grids(probs)
    out = vup.batched_outputs(grids, dds)
    for r in range(10):
        vup.propagate_batched(grids, dds, precision, out=out)
        assert vup.vup_batched_report()["source"] != 0, r  # a plan of its own
        for g in grids:
            g.sync()
        if r in (0, 4, 9):
            for p, raw, h in zip(probs, *out):
                _check(p, raw, h, precision)
        vup.propagate_batched(grids, dds, precision, out=out)
        assert vup.vup_batched_report()["source"] == 0, r  # the same call again replays it
        for g in grids if r % 2 else reversed(grids):
            g.close()
        # other models, so that what a stale graph left behind would show
        for p in probs:
            p.theta = (1.0 + 0.7 * (r + 1),)
        grids = _grids(probs)
    for g in grids:
        g.close()


def test_callers_graph_outlives_the_plans_of_other_batches():
    """A batch captured into a caller's graph, then more other batches than plans are
    kept for: the graph still replays the batch."""
    import torch
    from paper_1908_11246_gb300 import vup
    probs = I.oscillator_batch(31, n_inst=3, side=(40, 150), kk=(64, 500), n_bins=50)
    dds = [vup.densities_to_device(p.dens) for p in probs]
    grids = _grids(probs)
    out = vup.batched_outputs(grids, dds)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    vup.propagate_batched(grids, dds, "fp32", out=out, stream=s)
    s.synchronize()
    want = [t.clone() for t in out[0] + out[1]]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        vup.propagate_batched(grids, dds, "fp32", out=out, stream=s)
    others = [vup.batched_outputs(grids, dds) for _ in range(12)]  # 12 batches: other output buffers
    for _ in range(2):
        for o in others:
            vup.propagate_batched(grids, dds, "fp32", out=o)
    torch.cuda.synchronize()
    for t in out[0] + out[1]:
        t.fill_(-1)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(want, out[0] + out[1]):
        assert torch.equal(a, b)
    del graph
    for g in grids:
        g.close()
