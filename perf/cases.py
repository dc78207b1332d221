"""The work a user of the library has it do, as measured cases.

A case is one pass of one entry point (or of the few calls that belong
together) at one size.  ``prepare`` makes what a program holds before the
call -- the grid, usually with its model matrix, and the densities on the
device -- and ``run`` makes the calls.  ``exact`` gives the same outputs from
the definitions in double precision with plain torch.

Kinds of case (``case["kind"]``):

* ``line``       1-D grid in FP64: moments and histograms, with the IPSA
                 Jacobian where ``grad`` is set.
* ``plane``      2-D product Gaussians through ``Grid.propagate``.  ``model``
                 says what happens to the model in a pass: ``kept`` (one model
                 serves many sets of densities), ``new`` (every pass evaluates
                 the model anew: a parameter study) or ``supplied`` (every
                 pass hands over outputs that the user's own model computed).
* ``gradient``   ``vup_propagate_ipsa``: new model, forward pass and the vector-
                 Jacobian product of one set of densities in one call.
* ``autograd``   ``vup_moments`` inside a torch graph, forward and backward.
* ``volume``     3-D grid, each axis Gaussian, uniform or truncated normal.
* ``weights``    the input probability matrix given explicitly.
* ``posterior``  posterior means of the inputs per output bin.
* ``batch``      many small uneven instances in one batched call.
* ``study``      the sensitivity study of Sec. 5.3: model, propagation,
                 estimated values, deviation moments, IPSA matrix and the
                 marginalised vector.

Sizes are those of ``inputs.config`` / ``bench.py`` or generic ragged ones.
"""
import math

import numpy as np
import torch

from paper_1908_11246_gb300 import vup
from paper_1908_11246_gb300.autograd import vup_moments

GAUSS, UNIFORM, TRUNCNORM = 0, 1, 2
SIN_QUAD_1D, SIN_SIN2_2D, MIXED_3D, OSCILLATOR_2D, EXAMPLE_2D = 1, 2, 3, 4, 5
PI = math.pi
J = 4


def listed():
    return [
        # the smallest call in use: one axis, FP64 throughout
        dict(name="line_fp64", kind="line", n0=4096, K=256, B=64, grad=False),
        # a few hundred measurement locations against a model that is kept: latency and launches
        dict(name="plane_query", kind="plane", n0=200, n1=328, K=225, B=256, precision="bf16x3", model="kept"),
        # the timing experiment of Sec. 4.1 at full size: the model changes from pass to pass
        dict(name="plane_new_model", kind="plane", n0=1024, n1=1024, K=16384, B=256, precision="bf16x3", model="new"),
        # one model, set after set of densities, odd sizes
        dict(name="plane_kept_ragged", kind="plane", n0=1021, n1=613, K=9001, B=100, precision="bf16x3", model="kept"),
        # a user's own model evaluated elsewhere, in the precision without split products
        dict(name="plane_supplied_fp32", kind="plane", n0=900, n1=1100, K=3000, B=513, precision="fp32",
             model="supplied"),
        # the largest: forward pass and sensitivities of a 256 x 256 field of locations on a fine grid
        dict(name="gradient_field", kind="gradient", n0=2048, n1=2048, K=65536, B=256, precision="bf16x3"),
        # fitting: moments inside a torch graph, forward and backward in FP32
        dict(name="autograd_fp32", kind="autograd", n0=500, n1=400, K=2000, B=64, precision="fp32"),
        # three inputs with mixed densities
        dict(name="volume_mixed", kind="volume", n0=128, n1=128, n2=128, K=16384, B=512, precision="bf16x3",
             model="kept"),
        # input probabilities that are not product densities: the matrix itself is streamed
        dict(name="weights_matrix", kind="weights", n0=1024, n1=1024, K=1024, B=256),
        # inversion: which inputs led to an output bin
        dict(name="posterior_means", kind="posterior", n0=1024, n1=1024, K=8192, B=256),
        # many uneven instances of a parametric response, called again on the same buffers
        dict(name="batch_oscillators", kind="batch", count=32, side_lo=32, side_hi=1024, K_lo=64, K_hi=8192, B=128,
             shapes=5, precision="bf16x3"),
        # the whole Sec. 5.3 example
        dict(name="study_example", kind="study", n0=1000, n1=1000, K=1000, B=1000, precision="bf16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cap_k(K, N, most):
    return max(1, min(K, int(most // N)))


def draw(rng):
    kind = rng.choice(["line", "plane", "plane", "plane", "gradient", "autograd", "volume", "weights", "posterior",
                       "batch", "study"])
    if kind == "line":
        return dict(kind=kind, n0=_log(rng, 200, 20000), K=_log(rng, 8, 2048), B=_log(rng, 16, 512),
                    grad=rng.random() < 0.5)
    if kind == "plane":
        n0, n1 = _log(rng, 64, 2048), _log(rng, 64, 2048)
        prec = rng.choice(["bf16x3", "bf16x3", "bf16x3", "tf32x3", "fp32"])
        return dict(kind=kind, n0=n0, n1=n1, K=_cap_k(_log(rng, 64, 32768), n0 * n1, 4e10), B=_log(rng, 16, 1024),
                    precision=prec, model=rng.choice(["kept", "new", "supplied"]))
    if kind == "gradient":
        n0, n1 = _log(rng, 128, 2048), _log(rng, 128, 2048)
        return dict(kind=kind, n0=n0, n1=n1, K=_cap_k(_log(rng, 256, 65536), n0 * n1, 1e11), B=_log(rng, 32, 512),
                    precision=rng.choice(["bf16x3", "bf16x3", "fp32"]))
    if kind == "autograd":
        n0, n1 = _log(rng, 64, 1024), _log(rng, 64, 1024)
        return dict(kind=kind, n0=n0, n1=n1, K=_cap_k(_log(rng, 64, 8192), n0 * n1, 4e9), B=64,
                    precision=rng.choice(["fp32", "bf16x3"]))
    if kind == "volume":
        n = [_log(rng, 32, 160) for _ in range(3)]
        return dict(kind=kind, n0=n[0], n1=n[1], n2=n[2], K=_cap_k(_log(rng, 256, 32768), n[0] * n[1] * n[2], 3.5e10),
                    B=_log(rng, 32, 1024), precision=rng.choice(["bf16x3", "bf16x3", "fp32"]),
                    model=rng.choice(["kept", "new"]))
    if kind == "weights":
        n0, n1 = _log(rng, 64, 2048), _log(rng, 64, 2048)
        return dict(kind=kind, n0=n0, n1=n1, K=_cap_k(_log(rng, 64, 4096), n0 * n1, 1.0e9), B=_log(rng, 16, 1024))
    if kind == "posterior":
        n0, n1 = _log(rng, 128, 2048), _log(rng, 128, 2048)
        return dict(kind=kind, n0=n0, n1=n1, K=_cap_k(_log(rng, 64, 16384), n0 * n1, 1.0e10), B=_log(rng, 16, 512))
    if kind == "batch":
        return dict(kind=kind, count=_log(rng, 4, 32), side_lo=32, side_hi=_log(rng, 128, 1024), K_lo=64,
                    K_hi=_log(rng, 512, 8192), B=_log(rng, 32, 256), shapes=rng.randrange(1 << 20),
                    precision=rng.choice(["bf16x3", "bf16x3", "fp32"]))
    n0, n1 = _log(rng, 300, 1500), _log(rng, 100, 1500)
    return dict(kind="study", n0=n0, n1=n1, K=_log(rng, 32, 4000), B=_log(rng, 100, 2000),
                precision=rng.choice(["bf16x3", "fp32"]))


# ------------------------------------------------------------------- inputs
def _domain(case):
    """(sizes, lower bounds, upper bounds, model id, theta) of the case's grid."""
    kind = case["kind"]
    if kind == "line":
        return (case["n0"],), (-5.0,), (5.0,), SIN_QUAD_1D, (1.0, 0.1)
    if kind == "volume":
        return (case["n0"], case["n1"], case["n2"]), (-PI,) * 3, (PI,) * 3, MIXED_3D, (7.0, 0.1)
    if kind == "study":
        return (case["n0"], case["n1"]), (-5.0, -1.5), (5.0, 1.5), EXAMPLE_2D, ()
    return (case["n0"], case["n1"]), (-PI,) * 2, (PI,) * 2, SIN_SIN2_2D, (1.0, 7.0)


def _densities(case, seed):
    """Density parameters [K][ndim] as numpy arrays, from the seed alone."""
    rng = np.random.default_rng([int(seed), 77])
    n, lo, hi, _, _ = _domain(case)
    K, nd = case["K"], len(n)
    kind = np.zeros((K, nd), np.uint8)
    mu, sigma, tlo, thi = np.zeros((K, nd)), np.ones((K, nd)), np.zeros((K, nd)), np.zeros((K, nd))
    for d in range(nd):
        r = hi[d] - lo[d]
        h = r / n[d]
        mu[:, d] = rng.uniform(lo[d] + 0.05 * r, hi[d] - 0.05 * r, size=K)
        if case["kind"] == "line":
            sigma[:, d] = np.exp(rng.uniform(math.log(0.05), math.log(0.5), size=K))
        elif case["kind"] == "posterior":
            # prior knowledge of the inputs: wide enough that every output bin has mass
            sigma[:, d] = rng.uniform(0.5, 1.0, size=K)
        elif case["kind"] == "study":
            if d == 0:
                mu[:, 0] = lo[0] + (np.arange(K) + 0.5) * (r / K)
                sigma[:, 0] = rng.uniform(0.45, 0.55)
            else:
                mu[:, 1] = 0.0
                sigma[:, 1] = 0.25
        elif case["kind"] == "volume":
            kind[:, d] = rng.integers(0, 3, size=K)
            s = rng.uniform(max(0.05, 1.1 * h), max(0.6, 2.2 * h), size=K)
            w = rng.uniform(max(0.1, 2.2 * h), max(1.0, 4.4 * h), size=K)
            sigma[:, d] = np.where(kind[:, d] == UNIFORM, w, s)
            tn = kind[:, d] == TRUNCNORM
            tlo[:, d] = np.where(tn, mu[:, d] - rng.uniform(0.5, 3.0, size=K) * s, 0.0)
            thi[:, d] = np.where(tn, mu[:, d] + rng.uniform(0.5, 3.0, size=K) * s, 0.0)
        else:
            sigma[:, d] = rng.uniform(0.02, 0.6, size=K)
    return dict(kind=kind, mu=mu, sigma=sigma, lo=tlo, hi=thi)


def _on_device(d):
    return {k: torch.as_tensor(v, device="cuda") for k, v in d.items()}


def _outputs_of_model(case):
    """y on the grid by torch, as a user's own model would give it."""
    n, lo, hi, model, theta = _domain(case)
    return _model(n, lo, hi, model, theta).contiguous()


def _instances(case):
    """(side, K, T) of each instance of a batch."""
    rng = np.random.default_rng([int(case["shapes"]), 5])
    out = []
    for _ in range(case["count"]):
        side = int(round(math.exp(rng.uniform(math.log(case["side_lo"]), math.log(case["side_hi"])))))
        K = int(round(math.exp(rng.uniform(math.log(case["K_lo"]), math.log(case["K_hi"])))))
        out.append((side, K, float(rng.uniform(1.0, 10.0))))
    return out


OSC_LO, OSC_HI = (0.5, 0.01), (5.0, 0.9)


def _batch_densities(case, seed):
    rng = np.random.default_rng([int(seed), 78])
    out = []
    for _, K, _ in _instances(case):
        kind, tlo, thi = np.zeros((K, 2), np.uint8), np.zeros((K, 2)), np.zeros((K, 2))
        mu, sigma = np.zeros((K, 2)), np.zeros((K, 2))
        for d in range(2):
            r = OSC_HI[d] - OSC_LO[d]
            mu[:, d] = rng.uniform(OSC_LO[d] + 0.05 * r, OSC_HI[d] - 0.05 * r, size=K)
            sigma[:, d] = rng.uniform(0.02, 0.2, size=K) * r
        out.append(dict(kind=kind, mu=mu, sigma=sigma, lo=tlo, hi=thi))
    return out


def _weight_matrix(case, seed):
    """[K][N] FP32: normalised product Gaussians on the grid, each point's
    weight moved by up to 20 % (no longer a product)."""
    n, lo, hi, _, _ = _domain(case)
    w = _factors(n, lo, hi, _on_device(_densities(case, seed)))
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    K, N = case["K"], n[0] * n[1]
    W = torch.empty((K, N), dtype=torch.float32, device="cuda")
    w0, w1 = w[0].float(), w[1].float()
    step = max(1, (1 << 27) // N)
    for a in range(0, K, step):
        b = min(K, a + step)
        p = (w0[:, a:b].t()[:, :, None] * w1[:, a:b].t()[:, None, :]).reshape(b - a, N)
        W[a:b] = p * (0.8 + 0.4 * torch.rand((b - a, N), generator=g, device="cuda"))
    return W


def _grad_seed(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 2)
    return torch.randn((case["K"], J), generator=g, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        grids, dens = [], [_on_device(d) for d in _batch_densities(case, seed)]
        for side, _, T in _instances(case):
            g = vup.Grid((side, side), OSC_LO, OSC_HI)
            g.eval_model(OSCILLATOR_2D, (T,), case["B"], J)
            grids.append(g)
        raws, hists = vup.batched_outputs(grids, dens)
        call = vup.BatchedArgs([g.h for g in grids], [vup.make_densities(d) for d in dens], raws, hists)
        return dict(case=case, grids=grids, dens=dens, out=(raws, hists), call=call)
    n, lo, hi, model, theta = _domain(case)
    g = vup.Grid(n, lo, hi)
    st = dict(case=case, grid=g)
    if kind == "weights":
        st["W"] = _weight_matrix(case, seed)
    else:
        st["dens"] = _on_device(_densities(case, seed))
    if case.get("model") == "supplied":
        st["y"] = _outputs_of_model(case)
    elif case.get("model") != "new" and kind not in ("gradient", "study"):
        g.eval_model(model, theta, case["B"], J)
    if kind == "gradient":
        st["seed"] = _grad_seed(case, seed)
    if kind == "autograd":
        st["seed"] = _grad_seed(case, seed)
        st["dens"]["mu"].requires_grad_(True)
        st["dens"]["sigma"].requires_grad_(True)
    return st


# --------------------------------------------------------------------- calls
def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "batch":
        st["call"](vup.PRECISIONS[case["precision"]])
        return dict(raw=st["out"][0], hist=st["out"][1])
    g = st["grid"]
    K = case["K"]
    _, _, _, model, theta = _domain(case)
    if kind == "line":
        raw, cen, hist = g.propagate(st["dens"], "fp64")
        out = dict(raw=raw, central=cen, hist=hist)
        if case["grad"]:
            out["dmu"], out["dsigma"] = g.ipsa(st["dens"], "fp64")
        return out
    if kind in ("plane", "volume"):
        if case["model"] == "new":
            g.eval_model(model, theta, case["B"], J)
        elif case["model"] == "supplied":
            g.set_outputs(st["y"], case["B"], J)
        raw, cen, hist = g.propagate(st["dens"], case["precision"])
        return dict(raw=raw, central=cen, hist=hist)
    if kind == "gradient":
        g.eval_model(model, theta, case["B"], J)
        raw = torch.empty((K, J), dtype=torch.float64, device="cuda")
        cen = torch.empty((K, J), dtype=torch.float64, device="cuda")
        hist = torch.empty((K, case["B"]), dtype=torch.float32, device="cuda")
        dmu = torch.empty((K, 2), dtype=torch.float32, device="cuda")
        dsigma = torch.empty((K, 2), dtype=torch.float32, device="cuda")
        vup.vup_propagate_ipsa(g.h, vup.make_densities(st["dens"]), vup.PRECISIONS[case["precision"]], raw, cen, hist,
                               dmu, dsigma, st["seed"])
        return dict(raw=raw, central=cen, hist=hist, dmu=dmu, dsigma=dsigma)
    if kind == "autograd":
        d = st["dens"]
        d["mu"].grad = d["sigma"].grad = None
        raw = vup_moments(g, d, case["precision"])
        raw.backward(st["seed"])
        return dict(raw=raw.detach(), dmu=d["mu"].grad, dsigma=d["sigma"].grad)
    if kind == "weights":
        raw = torch.empty((K, J), dtype=torch.float64, device="cuda")
        hist = torch.empty((K, case["B"]), dtype=torch.float32, device="cuda")
        vup.vup_propagate_weights(g.h, st["W"], raw, hist)
        return dict(raw=raw, hist=hist)
    if kind == "posterior":
        hist = torch.empty((K, case["B"]), dtype=torch.float32, device="cuda")
        post = torch.empty((K, case["B"], 2), dtype=torch.float32, device="cuda")
        vup.vup_posterior_means(g.h, vup.make_densities(st["dens"]), hist, post)
        return dict(hist=hist, post=post)
    # study
    g.eval_model(model, theta, case["B"], J)
    raw, cen, hist = g.propagate(st["dens"], case["precision"])
    y = torch.empty(K, dtype=torch.float64, device="cuda")
    dev = torch.empty((K, J), dtype=torch.float64, device="cuda")
    mat = torch.empty((K, case["B"]), dtype=torch.float32, device="cuda")
    glob = torch.empty(case["B"], dtype=torch.float64, device="cuda")
    vup.vup_model_at(g.h, st["dens"]["mu"], y)
    vup.vup_deviation_moments(g.h, raw, y, dev)
    vup.vup_ipsa_matrix(g.h, hist, y, case["B"], -STUDY_SPAN, STUDY_SPAN, mat)
    vup.vup_sa_fields(mat, 0.9, global_=glob)
    return dict(raw=raw, central=cen, hist=hist, estimate=y, deviation=dev, matrix=mat, marginal=glob)


# deviations of the Sec. 5.3 example stay within twice its output range
STUDY_SPAN = 40.0


# ---------------------------------------------------------------------- work
PRODUCTS = {"fp64": 1, "fp32": 1, "bf16x3": 3, "tf32x3": 3}


def work(case):
    """Inputs read and outputs written once; the operations of the separable
    moment contraction (2 J per distribution-point, times the products that
    the chosen precision splits each into), or one multiply-add per
    distribution-point where there are no moments."""
    kind = case["kind"]
    if kind == "batch":
        bytes_ = flops = 0.0
        for side, K, _ in _instances(case):
            bytes_ += 4.0 * side * side + K * (2 * 33 + 8 * J + 4 * case["B"])
            flops += 2.0 * J * PRODUCTS[case["precision"]] * K * side * side
        return dict(bytes=bytes_, flops=flops)
    n = _domain(case)[0]
    N, nd, K, B = float(np.prod(n)), len(n), case["K"], case["B"]
    dens = K * nd * 33.0
    per = 2.0 * J * PRODUCTS[case.get("precision", "fp32")]
    if kind == "weights":
        return dict(bytes=4.0 * K * N + 12.0 * N + K * (8 * J + 4 * B), flops=2.0 * J * K * N)
    if kind == "posterior":
        return dict(bytes=4.0 * N + dens + K * B * 12.0, flops=2.0 * K * N)
    if kind == "autograd":
        return dict(bytes=8.0 * N + 2 * dens + K * (16 * J + 32), flops=3 * per * K * N)
    out = K * (16.0 * J + 4 * B)
    if kind == "gradient":
        return dict(bytes=12.0 * N + dens + out + K * (8 * J + 16), flops=2 * per * K * N)
    if kind == "study":
        return dict(bytes=12.0 * N + dens + out + K * (8 + 8 * J + 4 * B) + 8 * B, flops=per * K * N)
    grad = 2 * K * nd * J * 4.0 if case.get("grad") else 0.0
    return dict(bytes=12.0 * N + dens + out + grad, flops=per * K * N * (1 + 2 * bool(case.get("grad"))))


# --------------------------------------------------------------------- exact
def _axes(n, lo, hi):
    return [lo[d] + (torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * ((hi[d] - lo[d]) / n[d])
            for d in range(len(n))]


def _model(n, lo, hi, model, theta):
    x = _axes(n, lo, hi)
    if model == SIN_QUAD_1D:
        return theta[0] * torch.sin(x[0]) + theta[1] * x[0] * x[0]
    if model == SIN_SIN2_2D:
        s = torch.sin(x[1])
        return theta[0] * torch.sin(x[0])[:, None] + (theta[1] * (s * s))[None, :]
    if model == EXAMPLE_2D:
        return (x[0] * x[0] + 5.0 * torch.sin(3.0 * x[0]))[:, None] + x[1][None, :]
    if model == OSCILLATOR_2D:
        w, z = x[0][:, None], x[1][None, :]
        return torch.exp(-z * w * theta[0]) * torch.cos(w * torch.sqrt(1.0 - z * z) * theta[0])
    s0, s1 = torch.sin(x[0]), torch.sin(x[1])
    return (s0[:, None, None] + (theta[0] * (s1 * s1))[None, :, None] +
            theta[1] * (x[2] ** 4)[None, None, :] * s0[:, None, None])


def _bins(y, B):
    lo, hi = y.min(), y.max()
    return torch.clamp(torch.floor((y - lo) / (hi - lo) * B), 0, B - 1).to(torch.int64)


def _factors(n, lo, hi, d):
    """Per axis the normalised factors [n_d][K] in double precision."""
    out = []
    for a, x in enumerate(_axes(n, lo, hi)):
        mu, sg, kind = d["mu"][:, a], d["sigma"][:, a], d["kind"][:, a]
        dx = x[:, None] - mu[None, :]
        u = dx / sg
        gauss = torch.exp(-0.5 * (u * u - (u * u).min(0).values))
        inside = (x[:, None] >= d["lo"][:, a]) & (x[:, None] <= d["hi"][:, a])
        g = torch.where(kind == GAUSS, gauss, torch.zeros_like(gauss))
        g = torch.where(kind == UNIFORM, (dx.abs() <= 0.5 * sg).double(), g)
        if bool((kind == TRUNCNORM).any()):
            v = torch.where(inside, -0.5 * u * u, torch.full_like(u, -math.inf))
            v = torch.exp(v - v.max(0).values)
            g = torch.where(kind == TRUNCNORM, v, g)
        out.append(g / g.sum(0))
    return out


def _rest(w):
    """Products of all axes' factors but the last, [rows][K]."""
    r = w[0]
    for f in w[1:-1]:
        r = (r[:, None, :] * f[None, :, :]).reshape(-1, r.shape[1])
    return r


def _exact_hist(b, w, B):
    """H[K][B] by sums over stretches of one bin along the last axis."""
    n_last, K = w[-1].shape
    if len(w) == 1:
        H = torch.zeros((B, K), dtype=torch.float64, device="cuda")
        return H.index_add_(0, b, w[0]).t().contiguous()
    if len(w) == 2:  # the axis with fewer stretches as the last one
        cut = [int((b[1:] != b[:-1]).sum()), int((b[:, 1:] != b[:, :-1]).sum())]
        if cut[0] < cut[1]:
            b, w = b.t(), [w[1], w[0]]
            n_last = w[-1].shape[0]
    rows = b.reshape(-1, n_last)
    new = torch.ones_like(rows, dtype=torch.bool)
    new[:, 1:] = rows[:, 1:] != rows[:, :-1]
    r_id, start = torch.nonzero(new, as_tuple=True)
    end = torch.empty_like(start)
    end[:-1] = torch.where(r_id[1:] == r_id[:-1], start[1:], torch.full_like(start[1:], n_last))
    end[-1] = n_last
    bb = rows[r_id, start]
    H = torch.zeros((B, K), dtype=torch.float64, device="cuda")
    step_k = max(1, (1 << 25) // (w[0].shape[0] + n_last))
    for k0 in range(0, K, min(K, max(256, step_k))):
        k1 = min(K, k0 + min(K, max(256, step_k)))
        P = torch.zeros((n_last + 1, k1 - k0), dtype=torch.float64, device="cuda")
        torch.cumsum(w[-1][:, k0:k1], 0, out=P[1:])
        wk = [f[:, k0:k1].contiguous() for f in w[:-1]]
        m = max(1024, (1 << 27) // (k1 - k0))
        for s in range(0, r_id.numel(), m):
            t = slice(s, s + m)
            D = P[end[t]] - P[start[t]]
            if len(wk) == 1:
                D *= wk[0][r_id[t]]
            else:
                n1 = wk[1].shape[0]
                D *= wk[0][torch.div(r_id[t], n1, rounding_mode="floor")]
                D *= wk[1][r_id[t] % n1]
            H[:, k0:k1].index_add_(0, bb[t], D)
    return H.t().contiguous()


def _exact_raw(y, w):
    """Raw moments [K][J]."""
    out = []
    for j in range(1, J + 1):
        z = y ** j
        if len(w) == 1:
            out.append(z @ w[0])
        elif len(w) == 2:
            out.append(((z @ w[1]) * w[0]).sum(0))
        else:
            acc = 0.0
            for a in range(z.shape[0]):
                acc = acc + ((z[a] @ w[2]) * w[1]).sum(0) * w[0][a]
            out.append(acc)
    return torch.stack(out, 1)


def _central(raw, y, w):
    """Central moments from moments about the middle of the output range."""
    c = 0.5 * (y.min() + y.max())
    s = _exact_raw(y - c, w)
    m, s2, s3, s4 = s[:, 0], s[:, 1], s[:, 2], s[:, 3]
    return torch.stack([raw[:, 0], s2 - m * m, s3 - 3 * m * s2 + 2 * m ** 3,
                        s4 - 4 * m * s3 + 6 * m * m * s2 - 3 * m ** 4], 1)


def _exact_ipsa(case, y, w, d):
    """d raw_j / d mu and d sigma, [K][ndim][J] each."""
    n, lo, hi, _, _ = _domain(case)
    K, nd = w[0].shape[1], len(n)
    x = _axes(n, lo, hi)
    raw = _exact_raw(y, w)
    dmu = torch.zeros((K, nd, J), dtype=torch.float64, device="cuda")
    dsg = torch.zeros_like(dmu)
    for a in range(nd):
        dx = x[a][:, None] - d["mu"][:, a]
        sg = d["sigma"][:, a]
        ws = [w[a] * (dx / sg ** 2), w[a] * (dx * dx / sg ** 3)]
        bar = [v.sum(0) for v in ws]
        for j in range(1, J + 1):
            z = y ** j
            t = z[:, None].expand(-1, K) if nd == 1 else (z @ w[1] if a == 0 else z.t() @ w[0])
            for v, b, out in ((ws[0], bar[0], dmu), (ws[1], bar[1], dsg)):
                out[:, a, j - 1] = (t * v).sum(0) - b * raw[:, j - 1]
    return dmu, dsg


def _exact_batch(case, seed):
    raws, hists = [], []
    for (side, _, T), d in zip(_instances(case), _batch_densities(case, seed)):
        n = (side, side)
        y = _model(n, OSC_LO, OSC_HI, OSCILLATOR_2D, (T,))
        w = _factors(n, OSC_LO, OSC_HI, _on_device(d))
        raws.append(_exact_raw(y, w))
        hists.append(_exact_hist(_bins(y, case["B"]), w, case["B"]))
    return dict(raw=raws, hist=hists)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    n, lo, hi, model, theta = _domain(case)
    B = case["B"]
    y = _model(n, lo, hi, model, theta)
    b = _bins(y, B)
    if kind == "weights":
        W = _weight_matrix(case, seed)
        flat, fb = y.reshape(-1), b.reshape(-1)
        raw, hist = [], []
        step = max(1, (1 << 27) // flat.numel())
        for a in range(0, W.shape[0], step):
            w = W[a:a + step].double()
            raw.append(torch.stack([w @ flat ** j for j in range(1, J + 1)], 1))
            h = torch.zeros((B, w.shape[0]), dtype=torch.float64, device="cuda")
            hist.append(h.index_add_(0, fb, w.t().contiguous()).t())
        return dict(raw=torch.cat(raw), hist=torch.cat(hist))
    d = _on_device(_densities(case, seed))
    w = _factors(n, lo, hi, d)
    if kind == "posterior":
        x = _axes(n, lo, hi)
        H = _exact_hist(b, w, B)
        post = [_exact_hist(b, [w[0] * x[0][:, None], w[1]], B), _exact_hist(b, [w[0], w[1] * x[1][:, None]], B)]
        none = torch.zeros_like(H)  # bins that no grid point falls into
        return dict(hist=H, post=torch.stack([torch.where(H > 0, p / H, none) for p in post], 2))
    raw = _exact_raw(y, w)
    if kind in ("gradient", "autograd", "line") and (kind != "line" or case["grad"]):
        dmu, dsg = _exact_ipsa(case, y, w, d)
        if kind != "line":
            s = _grad_seed(case, seed)[:, None, :]
            dmu, dsg = (dmu * s).sum(2), (dsg * s).sum(2)
        if kind == "autograd":
            return dict(raw=raw, dmu=dmu, dsigma=dsg)
        return dict(raw=raw, central=_central(raw, y, w), hist=_exact_hist(b, w, B), dmu=dmu, dsigma=dsg)
    hist = _exact_hist(b, w, B)
    out = dict(raw=raw, central=_central(raw, y, w), hist=hist)
    if kind != "study":
        return out
    mu = d["mu"]
    est = mu[:, 0] ** 2 + 5.0 * torch.sin(3.0 * mu[:, 0]) + mu[:, 1]
    m = [torch.ones_like(est)] + [raw[:, j] for j in range(J)]
    out["deviation"] = torch.stack([sum(math.comb(j, i) * m[i] * (-est) ** (j - i) for i in range(j + 1))
                                    for j in range(1, J + 1)], 1)
    width = 2 * STUDY_SPAN / B
    centre = y.min() + (torch.arange(B, dtype=torch.float64, device="cuda") + 0.5) * ((y.max() - y.min()) / B)
    to = torch.floor((centre[None, :] - est[:, None] + STUDY_SPAN) / width).clamp(0, B - 1).to(torch.int64)
    mat = torch.zeros_like(hist).scatter_add_(1, to, hist)
    out.update(estimate=est, matrix=mat, marginal=mat.mean(0))
    return out
