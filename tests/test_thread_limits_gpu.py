"""Two host threads, each with grids and a stream of its own, whose kernels want
different amounts of shared memory past the default limit: the limit belongs to
a kernel, so a thread that set its own size could lower it between another's
setting and launch.  Every call must succeed and give what it gives alone."""
import ctypes
import threading

import numpy as np
import pytest
import torch

from paper_1908_11246_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_1908_11246_gb300 import build
    build.build()


def _setup(n, K, precision, B=32):
    from paper_1908_11246_gb300 import vup
    nd = len(n)
    rng = np.random.default_rng(n[0] + K)
    dens = I.random_densities(rng, K, (-1.0,) * nd, (1.0,) * nd, sig=(0.4, 1.0), margin=0.2)
    y = np.cumsum(np.abs(rng.standard_normal(n)), axis=0)
    g = vup.Grid(n, (-1.0,) * nd, (1.0,) * nd)
    y = torch.as_tensor(y, device="cuda")
    g.set_outputs(y, B)
    return g, y, vup.densities_to_device(dens), precision, B


@pytest.mark.parametrize("sizes, K, precision, new_model, calls", [
    (((5300,), (6100,)), 700, "fp64", False, 20000),            # one CTA per density: all of the axis' points
    (((11500, 3), (16000, 3)), 64, "fp32", True, 1000),         # class lists of long axes, tiles of their parts
    (((250, 260), (330, 390)), 300, "fp32", False, 5000),      # tiles of unlike height
])
def test_two_threads_with_unlike_sizes(sizes, K, precision, new_model, calls):
    work = [_setup(n, K, precision) for n in sizes]
    want = []
    for g, y, dd, prec, B in work:
        want.append([t.clone() for t in g.propagate(dd, prec, central=False)[::2]])
        g.sync()
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(work))

    def run(i):
        from paper_1908_11246_gb300 import vup
        g, y, dd, prec, B = work[i]
        try:
            s = torch.cuda.Stream()
            raw, hist = (torch.zeros_like(t) for t in want[i])
            torch.cuda.synchronize()
            # nothing but the library's calls in the loop, so that they overlap
            lib, d = vup.lib(), vup.make_densities(dd)
            p, st = vup._ptr, vup._stream(s)
            args = (g.h, ctypes.byref(d), vup.PRECISIONS[prec], p(raw), None, p(hist), st)
            outs = (g.h, p(y), B, 4, st)
            start.wait()
            for c in range(calls):
                bad = (lib.vup_set_outputs(*outs) if new_model else 0) or lib.vup_propagate(*args)
                if bad:
                    errors.append((sizes[i], c, vup.vup_status_string(bad), vup.vup_last_error_detail()))
                    return
                if c % 50 == 49:
                    s.synchronize()
            s.synchronize()
            same = [torch.equal(a, b) for a, b in zip(want[i], (raw, hist))]
            if not all(same):
                errors.append((sizes[i], same))
        except Exception as e:  # reported by the main thread
            errors.append((sizes[i], repr(e)))

    threads = [threading.Thread(target=run, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for g, *_ in work:
        g.close()
