"""The work that users of this framework have it do, as cases that can be timed and checked.

A muSR analysis uploads the positron histograms of a run once and then asks for the cost and
its gradient many times: one parameter vector at a time (a minimiser's steps), some tens at a
time (curvature estimates, multi-start and parameter scans), or through the fit, the parameter
errors and the fit server that are built on those.  The other workload is the open-boundary
particle-mesh Poisson solve.  Every case goes through the package's public entry points
(``binding``, ``autograd``).

``listed()`` names twelve such calls, ``draw(rng)`` gives others of the same ranges,
``prepare`` makes what the caller holds beforehand (histograms drawn from the model with
Poisson statistics, the configured context, the parameter vectors), ``run`` is one call, and
``exact`` the same result from plain 64-bit torch or numpy.
"""
import math

import numpy as np
import torch

from paper_1509_07685_gb300 import autograd as A
from paper_1509_07685_gb300 import binding as B

TAU_US = 2.197019
SPAN_NS = 12800.0  # length of a run's time window
DEV = "cuda:0"
MODES = {"chi2": B.MUSR_CHI2, "mle": B.MUSR_MLE}
PRECISIONS = {"split": B.MUSR_SPLIT, "fp64": B.MUSR_FP64}


def listed():
    return [
        # A minimiser's step on the smallest run: one detector, int32 counts as the data
        # acquisition writes them.  Latency of one launch and its copies.
        dict(name="one_detector_step", call="eval", theory="tf1", nhist=1, nbins=16384, dtype="int32",
             precision="split", mode="mle", nvec=1, grad=True, t0="same"),
        # The same step of an ordinary global fit: 8 detectors, 28 parameters.
        dict(name="global_fit_step", call="eval", theory="tf2", nhist=8, nbins=65536, dtype="fp32",
             precision="split", mode="mle", nvec=1, grad=True, t0="same"),
        # The whole fit of that run (native BFGS): some tens of steps and a batch for the curvature.
        dict(name="global_fit", call="fit", theory="tf2", nhist=8, nbins=65536, dtype="fp32",
             precision="split", mode="mle", t0="same"),
        # A multi-start batch on the 16-detector instrument, 66 parameters, host arrays in and out.
        dict(name="multistart_16", call="eval", theory="tf", nhist=16, nbins=81920, dtype="fp32",
             precision="split", mode="chi2", nvec=64, grad=True, t0="same"),
        # The largest run (64 detectors, fine bins, low counts) at 64 trial points, arrays on the GPU.
        dict(name="large_run_batch", call="eval_device", theory="tf2kt", nhist=64, nbins=1 << 20, dtype="fp32",
             precision="split", mode="mle", nvec=64, grad=True, t0="same"),
        # The full-precision step that polishes or checks a fit, FP64 histograms.
        dict(name="global_fit_step_fp64", call="eval", theory="tf2", nhist=8, nbins=65536, dtype="fp64",
             precision="fp64", mode="mle", nvec=1, grad=True, t0="same"),
        # A likelihood map: the cost alone at 1000 points of one detector in full precision.
        dict(name="cost_scan_fp64", call="eval", theory="tf1", nhist=1, nbins=16384, dtype="int32",
             precision="fp64", mode="mle", nvec=1000, grad=False, t0="same"),
        # Parameter errors after the fit: the full-precision Gauss-Newton matrix.
        dict(name="errors_fp64", call="errors", theory="tf2", nhist=8, nbins=65536, dtype="fp32",
             precision="fp64", mode="mle", t0="same"),
        # Asymmetry data of 7 detector pairs, a rebinned odd length, each pair with its own time zero.
        dict(name="asymmetry_odd", call="eval", theory="asym", nhist=7, nbins=30011, dtype="fp32",
             precision="split", mode="chi2", nvec=24, grad=True, t0="each"),
        # A zero-field run in fluctuating fields, one step through torch's autograd (the table of
        # the relaxation is solved in every step).
        dict(name="fluctuating_step", call="autograd", theory="dkt", nhist=16, nbins=81920, dtype="fp32",
             precision="split", mode="mle", nvec=1, grad=True, t0="same"),
        # The space-charge solve of a tracking step, arrays on the GPU.
        dict(name="space_charge", call="poisson", nx=256, ny=256, nz=128, precision="fp64"),
        # A beam time's worth of mixed fits handed to the server at once.
        dict(name="served_fits", call="serve", fits=24, max_hist=64, max_bins=262144, precision="split"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes over the ranges of the listed ones, odd ones among them."""
    call = rng.choice(["eval", "eval", "eval", "eval_device", "autograd", "errors", "poisson", "fit"])
    if call == "poisson":
        return dict(call=call, nx=_log(rng, 16, 256), ny=_log(rng, 16, 256), nz=_log(rng, 16, 128),
                    precision=rng.choice(["fp64", "split"]))
    precision = rng.choice(["split", "split", "fp64"])
    if call == "fit":
        return dict(call=call, theory=rng.choice(["tf2", "tf"]), nhist=_log(rng, 2, 16), nbins=_log(rng, 16384, 131072),
                    dtype="fp32", precision=precision, mode="mle", t0="same")
    theory = rng.choice(["tf1", "tf2", "tf", "zf", "tf2kt", "asym", "dkt", "strexp", "bessel"])
    if call == "errors" and theory in ("asym", "dkt", "strexp", "bessel"):
        precision = "fp64"  # the split path gives no such products for these (or only approximately: dkt)
    nhist, nbins = (1 if theory == "tf1" else _log(rng, 1, 64)), _log(rng, 4096, 262144)
    most = (2.0e7 if precision == "fp64" else 1.0e9) / (nhist * nbins)  # (histogram, bin) pairs of one call
    nvec = 1 if call in ("autograd", "errors") else _log(rng, 1, max(1, min(1000 if theory == "tf1" else 64, most)))
    if call == "errors":
        nhist = min(nhist, 12)
        nbins = min(nbins, 65536)
    dtype = rng.choice(["int32", "fp32", "fp64"] if call == "eval" else ["fp32", "fp64"])
    mode = "chi2" if theory == "asym" else rng.choice(["chi2", "mle"])
    return dict(call=call, theory=theory, nhist=nhist, nbins=nbins, dtype=dtype, precision=precision, mode=mode,
                nvec=nvec, grad=call != "eval" or rng.random() < 0.75, t0=rng.choice(["same", "each"]))


# ---------------------------------------------------------------------------------------------
# Theories: term lists, parameter maps, truths
# ---------------------------------------------------------------------------------------------

def _theory(kind, H):
    """(terms, map [H][nslots], constants, truth, names) of a theory on H histograms."""
    ph = [360.0 * j / max(H, 8) for j in range(H)]
    if kind == "tf1":
        terms = [[("AMP", (2,)), ("EXP", (3,)), ("TFCOS", (4, 5))]]
        names, truth = ["A", "lambda", "nu"], [0.25, 0.5, 5.0]
        own = [("N0", 300.0), ("Nbkg", 2.0), ("phi", None)]
        row = lambda b: [b, b + 1, 0, 1, 2, b + 2]  # noqa: E731
        consts = []
    elif kind in ("tf2", "tf2kt"):
        terms = [[("AMP", (2,)), ("EXP", (3,)), ("TFCOS", (4, 5))], [("AMP", (6,)), ("GAUSS", (7,)), ("TFCOS", (8, 5))]]
        names, truth = ["lambda", "sigma", "nu1", "nu2"], [0.5, 0.3, 5.0, 5.5]
        consts = [0.125, 0.125]
        row = lambda b: [b, b + 1, -1, 0, 2, b + 2, -2, 1, 3]  # noqa: E731
        own = [("N0", 300.0), ("Nbkg", 2.0), ("phi", None)]
        if kind == "tf2kt":  # low counts per bin
            terms, consts = terms + [[("AMP", (9,)), ("KT", (10,))]], consts + [0.05]
            names, truth = names + ["Delta"], truth + [0.3]
            row = lambda b: [b, b + 1, -1, 0, 2, b + 2, -2, 1, 3, -3, 4]  # noqa: E731
            own = [("N0", 2.0), ("Nbkg", 0.01), ("phi", None)]
    elif kind == "tf":
        terms, consts = [[("AMP", (2,)), ("GAUSS", (3,)), ("TFCOS", (4, 5))]], []
        names, truth = ["sigma", "nu"], [0.3, 10.0]
        own = [("N0", 300.0), ("Nbkg", 2.0), ("A", 0.22), ("phi", None)]
        row = lambda b: [b, b + 1, b + 2, 0, 1, b + 3]  # noqa: E731
    elif kind == "zf":
        terms, consts = [[("AMP", (2,)), ("KT", (3,)), ("EXP", (4,))]], []
        names, truth = ["A", "Delta", "lambda"], [0.25, 0.3, 0.1]
        own = [("N0", 300.0), ("Nbkg", 2.0)]
        row = lambda b: [b, b + 1, 0, 1, 2]  # noqa: E731
    elif kind == "dkt":
        terms, consts = [[("AMP", (2,)), ("DKT", (3, 4))]], []
        names, truth = ["A", "Delta", "nu_c"], [0.25, 0.4, 0.8]
        own = [("N0", 300.0), ("Nbkg", 2.0)]
        row = lambda b: [b, b + 1, 0, 1, 2]  # noqa: E731
    elif kind == "asym":  # scale 1 and baseline 0, a phase per pair
        terms, consts = [[("AMP", (2,)), ("GAUSS", (3,)), ("TFCOS", (4, 5))]], [1.0, 0.0]
        names, truth = ["A", "sigma", "nu"], [0.22, 0.4, 3.0]
        own = [("phi", None)]
        row = lambda b: [-1, -2, 0, 1, 2, b]  # noqa: E731
    elif kind == "strexp":
        terms, consts = [[("AMP", (2,)), ("STREXP", (3, 4))]], []
        names, truth = ["A", "lambda", "beta"], [0.25, 0.8, 0.5]
        own = [("N0", 300.0), ("Nbkg", 2.0)]
        row = lambda b: [b, b + 1, 0, 1, 2]  # noqa: E731
    elif kind == "bessel":
        terms, consts = [[("AMP", (2,)), ("BESSEL", (3, 4)), ("EXP", (5,))]], [0.0]
        names, truth = ["nu", "lambda"], [2.5, 0.3]
        own = [("N0", 300.0), ("Nbkg", 2.0), ("A", 0.22)]
        row = lambda b: [b, b + 1, b + 2, 0, -1, 1]  # noqa: E731
    else:
        raise ValueError(kind)
    rows, first = [], len(truth)
    names, truth = list(names), list(truth)
    for j in range(H):
        rows.append(row(first + len(own) * j))
        for n, v in own:
            names.append(n)
            truth.append(ph[j] if v is None else v)
    return terms, np.array(rows, np.int32), np.array(consts), np.array(truth), names


def _jitter(rng, truth, names, rel, nu_rel, phase):
    """A point near the truth as a fit meets it: frequencies from the run's FFT, phases in degrees."""
    x = truth.copy()
    for i, n in enumerate(names):
        if n.startswith("nu") and n != "nu_c":
            x[i] *= 1.0 + rng.uniform(-nu_rel, nu_rel)
        elif n == "phi":
            x[i] += rng.uniform(-phase, phase)
        else:
            x[i] *= 1.0 + rng.uniform(-rel, rel)
    return x


# ---------------------------------------------------------------------------------------------
# The model in 64-bit torch
# ---------------------------------------------------------------------------------------------

def _dkt(D, nu, span):
    """Strong-collision relaxation on a grid over [0, span]: (h, G, dG/dD, dG/dnu), FP64.  The
    renewal equation by the trapezoidal rule on h and h/2 and Richardson extrapolation."""
    K = int(min(max(math.ceil(span * max(abs(D), abs(nu), 0.05) / 0.008), 512), 4096))

    def solve(K):
        h = span / K
        t = h * np.arange(K + 1)
        u, e = (D * t) ** 2, np.exp(-nu * t)
        gg = np.exp(-0.5 * u)
        g = 1.0 / 3.0 + 2.0 / 3.0 * (1.0 - u) * gg
        f, fD, fN = g * e, 2.0 / 3.0 * D * t * t * gg * (u - 3.0) * e, -t * g * e
        a, b, c = 1.0 - 0.5 * nu * h, 1.0 + 0.5 * nu * h, nu * h
        G, GD, GN = (np.zeros(K + 1) for _ in range(3))
        G[0] = 1.0
        for k in range(1, K + 1):
            r = slice(k - 1, 0, -1)
            s = f[r] @ G[1:k]
            G[k] = (b * f[k] + c * s) / a
            GD[k] = (b * fD[k] + c * (fD[r] @ G[1:k] + f[r] @ GD[1:k])) / a
            GN[k] = (0.5 * h * (f[k] + G[k]) + b * fN[k] + h * s + c * (fN[r] @ G[1:k] + f[r] @ GN[1:k])) / a
        return h, G, GD, GN

    h, *c = solve(K)
    _, *f = solve(2 * K)
    return (h, *((4.0 * y[::2] - x) / 3.0 for x, y in zip(c, f)))


def _cubic(table, h, t):
    K = table.numel() - 1
    x = (t / h).clamp(min=0.0)
    i = (x.floor() - 1.0).clamp(0, K - 3)
    u, i = x - i, i.long()
    w = (-(u - 1) * (u - 2) * (u - 3) / 6, u * (u - 2) * (u - 3) / 2, -u * (u - 1) * (u - 3) / 2, u * (u - 1) * (u - 2) / 6)
    return sum(a * table[i + k] for k, a in enumerate(w))


def _asymmetry(terms, loc, t):
    """A(t) and its derivative by each local slot, broadcast over loc's histograms [H][nslots] and t [H or 1][B]."""
    total, ders = 0.0, {}
    one = bool((loc == loc[:1]).all(0).all())  # every slot the same: one row is enough
    col = lambda s: loc[:1, s:s + 1] if one or bool((loc[:, s] == loc[0, s]).all()) else loc[:, s:s + 1]  # noqa: E731
    for term in terms:
        f, df = [], []
        for kind, s in term:
            p = [col(q) for q in s]
            if kind == "AMP":
                v, d = p[0], [torch.ones_like(p[0])]
            elif kind == "EXP":
                v = torch.exp(-p[0] * t)
                d = [-t * v]
            elif kind == "GAUSS":
                v = torch.exp(-0.5 * (p[0] * t) ** 2)
                d = [-p[0] * t * t * v]
            elif kind == "KT":
                u = (p[0] * t) ** 2
                g = torch.exp(-0.5 * u)
                v, d = 1.0 / 3.0 + 2.0 / 3.0 * (1.0 - u) * g, [2.0 / 3.0 * p[0] * t * t * g * (u - 3.0)]
            elif kind == "TFCOS":
                x = p[0] * t + p[1] / 360.0
                r = 2.0 * math.pi * (x - torch.round(x))
                sn = torch.sin(r)
                v, d = torch.cos(r), [-2.0 * math.pi * t * sn, -2.0 * math.pi / 360.0 * sn]
            elif kind == "STREXP":
                x = (p[0] * t).clamp(min=1e-300)
                xb = x ** p[1]
                v = torch.exp(-xb)
                d = [-p[1] * xb / p[0] * v, -xb * torch.log(x) * v]
            elif kind == "BESSEL":
                x = 2.0 * math.pi * (p[0] * t + p[1] / 360.0)
                j1 = torch.special.bessel_j1(x)
                v, d = torch.special.bessel_j0(x), [-j1 * 2.0 * math.pi * t, -j1 * 2.0 * math.pi / 360.0]
            else:  # DKT: Delta and nu are shared
                h, *tab = _dkt(float(p[0][0, 0]), float(p[1][0, 0]), float(t.max()))
                v, *d = (_cubic(torch.from_numpy(y).to(t.device), h, t) for y in tab)
            f.append(v)
            df.append((s, d))
        prod = 1.0
        for v in f:
            prod = prod * v
        total = total + prod
        for m, (s, d) in enumerate(df):
            rest = 1.0
            for q, v in enumerate(f):
                rest = rest * v if q != m else rest
            for slot, dv in zip(s, d):
                ders[slot] = ders.get(slot, 0.0) + dv * rest
    return total, ders


def _model(terms, loc, t, envelope):
    """N and its local derivatives {slot: dN/dslot}."""
    a, da = _asymmetry(terms, loc, t)
    E = torch.exp(-t / TAU_US) if envelope else torch.ones_like(t)
    n0 = loc[:, 0:1]
    shape = E * ((1.0 + a) if envelope else a)
    ders = {s: n0 * E * d for s, d in da.items()}
    ders[0], ders[1] = shape, torch.ones_like(shape)
    return n0 * shape + loc[:, 1:2], ders


def _times(p, h):
    """Bin times of histograms h (a slice) and which bins are in the fit."""
    n = torch.arange(p["B"], dtype=torch.float64, device=DEV)[None, :]
    t0 = torch.from_numpy(p["t0"][h]).to(DEV)[:, None]
    if bool((t0 == t0[0]).all()):
        t0 = t0[:1]
    t = (n - t0) * (p["bw"] / 1000.0)
    return t, (t >= p["range"][0]) & (t <= p["range"][1])


def _local(p, x):
    m = torch.from_numpy(p["map"]).to(DEV).long()
    every = torch.cat([torch.from_numpy(np.asarray(x, np.float64)), torch.from_numpy(p["consts"])]).to(DEV)
    return m, every[torch.where(m >= 0, m, p["P"] - 1 - m)]


def _slices(p):
    step = max(1, int(2 ** 25 // p["B"]))
    return [slice(a, min(a + step, p["H"])) for a in range(0, p["H"], step)]


def _cost(p, x, mode, grad):
    """Value and gradient of the cost at one parameter vector, FP64."""
    m, loc = _local(p, x)
    value, g = 0.0, torch.zeros(p["P"], dtype=torch.float64, device=DEV)
    for h in _slices(p):
        t, inside = _times(p, h)
        N, ders = _model(p["terms"], loc[h], t, p["w"] is None)
        d = p["counts"][h].double()
        if mode == "chi2":
            w = p["w"][h] if p["w"] is not None else 1.0 / d.clamp(min=1.0)
            v, W = w * (d - N) ** 2, -2.0 * w * (d - N)
        else:
            safe = torch.where(d > 0, d, torch.ones_like(d))
            v = 2.0 * ((N - d) + torch.where(d > 0, d * torch.log(safe / N), torch.zeros_like(d)))
            W = 2.0 * (1.0 - d / N)
        value = value + (v * inside).sum()
        if grad:
            W = W * inside
            for s, dn in ders.items():
                col = (W * dn).sum(1)
                at = m[h, s]
                g.index_add_(0, at[at >= 0], col[at >= 0])
    return value, g


def _gauss_newton(p, x, mode):
    """Sum over bins of (d2 cost / dN2) J J^T, FP64."""
    m, loc = _local(p, x)
    out = torch.zeros(p["P"], p["P"], dtype=torch.float64, device=DEV)
    for j in range(p["H"]):
        h = slice(j, j + 1)
        t, inside = _times(p, h)
        N, ders = _model(p["terms"], loc[h], t, p["w"] is None)
        d = p["counts"][h].double()
        w = 2.0 * p["w"][h] if p["w"] is not None else 2.0 / d.clamp(min=1.0) if mode == "chi2" else 2.0 * d / (N * N)
        slots = [s for s in sorted(ders) if int(m[j, s]) >= 0]
        J = torch.cat([ders[s].expand(1, p["B"]) for s in slots])
        at = m[j, slots]
        local = (J * (w * inside)) @ J.T
        out.index_put_((at[:, None].expand_as(local), at[None, :].expand_as(local)), local, accumulate=True)
    return out


def _optimum(p, x0, mode):
    """The fit's result: the minimum of the cost near x0, by damped Gauss-Newton steps."""
    x, (f, g) = np.array(x0), _cost(p, x0, mode, True)
    for _ in range(40):
        H = _gauss_newton(p, x, mode)
        scale = H.diagonal().clamp(min=1e-300).rsqrt()
        step = (scale * torch.linalg.solve(H * scale[:, None] * scale, scale * g)).cpu().numpy()
        if float(g.cpu().numpy() @ step) < 1e-18 * float(f):
            break
        a = 1.0
        while a > 1e-4:
            fn, gn = _cost(p, x - a * step, mode, True)
            if float(fn) <= float(f) * (1.0 + 1e-14):
                break
            a *= 0.5
        x, f, g = x - a * step, fn, gn
    return x, f


# ---------------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------------

def _problem(theory, H, nbins, dtype, t0, seed):
    """A run: histograms with Poisson statistics of a model near the theory's truth."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(DEV).manual_seed(seed)
    terms, mp, consts, truth, names = _theory(theory, H)
    truth = _jitter(rng, truth, names, 0.05, 0.05, 10.0)
    bw = SPAN_NS / nbins if theory != "tf1" else 0.5 * 16384 / nbins
    dt = bw / 1000.0
    p = dict(H=H, B=nbins, P=truth.size, terms=terms, map=mp, consts=consts, truth=truth, names=names, bw=bw, w=None,
             t0=np.zeros(H) if t0 == "same" else rng.integers(5, 40, H).astype(np.float64), range=(0.5 * dt, nbins * dt))
    real = {"int32": torch.int32, "fp32": torch.float32, "fp64": torch.float64}[dtype]
    _, loc = _local(p, truth)
    if theory == "asym":  # forward and backward detectors, efficiency 0.85, a flat background of 3
        F, Bk, n0, eff, bkg = [], [], 400.0, 0.85, 3.0
        for h in _slices(p):
            t, _ = _times(p, h)
            a, _ = _asymmetry(terms, loc[h], t)
            live = torch.where(t >= 0, n0 * torch.exp(-t / TAU_US), torch.zeros_like(t))
            F.append(torch.poisson(live * (1.0 + a) + bkg, generator=gen).to(real))
            Bk.append(torch.poisson(eff * live * (1.0 - a) + bkg, generator=gen).to(real))
        p["pairs"] = (torch.cat(F), torch.cat(Bk))
        p["alpha"], p["bkg"] = np.full(H, 1.0 / eff), np.full(H, bkg)
    else:
        rows = []
        for h in _slices(p):
            t, _ = _times(p, h)
            N, _ = _model(terms, loc[h], t.clamp(min=0.0), True)
            N = torch.where(t >= 0, N, loc[h][:, 1:2].expand_as(N))
            rows.append(torch.poisson(N, generator=gen).to(real))
        p["counts"] = torch.cat(rows)
    return p


def _vectors(p, nvec, grad, seed):
    """Trial points: near the truth for a minimiser, spread by 20 % for a map of the cost."""
    rng = np.random.default_rng(seed + 1)
    if not grad:
        return p["truth"][None, :] * rng.uniform(0.8, 1.2, (nvec, p["P"]))
    return np.stack([_jitter(rng, p["truth"], p["names"], 0.02, 0.002, 5.0) for _ in range(nvec)])


def _exact_data(p):
    """Asymmetry and weights in FP64 from the pairs."""
    if "pairs" in p:
        F, Bk = (v.double() for v in p["pairs"])
        al = torch.from_numpy(p["alpha"]).to(DEV)[:, None]
        bk = torch.from_numpy(p["bkg"]).to(DEV)[:, None]
        f, b = F - bk, Bk - bk
        D = f + al * b
        ok = D > 0
        D = torch.where(ok, D, torch.ones_like(D))
        var = 4.0 * al * al * (b * b * F.clamp(min=1.0) + f * f * Bk.clamp(min=1.0)) / D ** 4
        p["counts"] = torch.where(ok, (f - al * b) / D, torch.zeros_like(D))
        p["w"] = torch.where(ok & (var > 0), 1.0 / torch.where(var > 0, var, torch.ones_like(var)), torch.zeros_like(D))
    return p


def _context(p, dtype):
    """A context on torch's stream, configured for the run; arrays of the GPU are lent to it."""
    ctx = B.Context(cuda_stream=torch.cuda.current_stream().cuda_stream)
    if "pairs" in p:
        F, Bk = (v.cpu().numpy() for v in p["pairs"])
        B.musr_upload_asymmetry(ctx.ctx, F, Bk, p["t0"], p["bw"], p["range"], p["alpha"], p["bkg"], p["bkg"])
    elif dtype == "int32" or len(set(p["t0"])) > 1 or p["B"] % 4:
        B.musr_upload_histograms(ctx.ctx, p["counts"].cpu().numpy(), p["t0"], p["bw"], p["range"])
    else:
        B.musr_upload_histograms_device(ctx.ctx, p["counts"].data_ptr(), B.MUSR_DTYPE_FP32 if dtype == "fp32" else B.MUSR_DTYPE_FP64,
                                        p["H"], p["B"], p["B"], p["t0"], p["bw"], p["range"])
    B.musr_set_theory(ctx.ctx, p["terms"])
    B.musr_set_map(ctx.ctx, p["map"], p["P"], p["consts"])
    ctx.P = p["P"]
    return ctx


def _served(case, seed):
    """The runs a server gets: sizes spread over their logarithm, three theories, both costs.  The
    sizes are the case's own (the same for every seed), the counts and start points the seed's."""
    sizes = np.random.default_rng(4)
    rng = np.random.default_rng(seed)
    got = []
    for i in range(case["fits"]):
        kind = ("tf1", "tf2", "zf")[i % 3]
        H = int(round(math.exp(sizes.uniform(0.0, math.log(case["max_hist"])))))
        nbins = int(round(math.exp(sizes.uniform(math.log(4096), math.log(case["max_bins"])))))
        p = _problem(kind, 1 if kind == "tf1" else H, nbins, "fp32", "same", int(rng.integers(1 << 30)))
        got.append((p, _jitter(rng, p["truth"], p["names"], 0.02, 0.002, 5.0), "mle" if i % 2 else "chi2"))
    return got


class _Request:
    """A fit as the server takes it."""

    def __init__(self, p):
        self.counts, self.t0, self.bin_width_ns, self.fit_range_us = p["counts"].cpu().numpy(), p["t0"], p["bw"], p["range"]
        self.terms, self.map, self.consts, self.nparams = p["terms"], p["map"], p["consts"], p["P"]


# ---------------------------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------------------------

def _density(case, seed):
    """A bunch's charge density with the noise of its macroparticles."""
    gen = torch.Generator(DEV).manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    axes = [((torch.arange(k, dtype=torch.float64, device=DEV) + 0.5) / k - 0.5) / s for k, s in zip(n, (0.12, 0.15, 0.2))]
    rate = 50.0 * torch.exp(-0.5 * (axes[0][:, None, None] ** 2 + axes[1][None, :, None] ** 2 + axes[2][None, None, :] ** 2))
    return torch.poisson(rate, generator=gen), (1.0e-3 * 96 / n[0], 1.1e-3 * 96 / n[1], 1.5e-3 * 96 / n[2])


def prepare(case, seed):
    s = dict(case=case, call=case["call"], precision=PRECISIONS[case["precision"]])
    if s["call"] == "poisson":
        rho, h = _density(case, seed)
        s["rho"], s["phi"] = rho, torch.empty_like(rho)
        s["solver"] = B.Poisson(tuple(rho.shape), h, s["precision"], cuda_stream=B.CUDA_STREAM_LEGACY)
        return s
    if s["call"] == "serve":
        s["server"] = B.Server(hbm_budget_bytes=2 << 30)
        s["fits"] = [(_Request(p), x0, MODES[m]) for p, x0, m in _served(case, seed)]
        return s
    p = _problem(case["theory"], case["nhist"], case["nbins"], case["dtype"], case["t0"], seed)
    s["mode"], s["grad"] = MODES[case["mode"]], case.get("grad", True)
    s["counts"] = p.get("counts")  # lent to the context
    s["ctx"] = _context(p, case["dtype"])
    s["x"] = _vectors(p, case.get("nvec", 1), s["grad"], seed)
    if s["call"] == "eval_device":
        s["d_x"] = torch.from_numpy(s["x"]).to(DEV)
        s["d_out"] = torch.empty(s["x"].shape[0], 1 + p["P"], dtype=torch.float64, device=DEV)
    if s["call"] == "autograd":
        s["t_x"] = torch.from_numpy(s["x"][0]).to(DEV).requires_grad_()
    return s


def run(s):
    call = s["call"]
    if call == "poisson":
        s["solver"].solve_device(s["rho"].data_ptr(), s["phi"].data_ptr())
        return s["phi"]
    if call == "serve":
        ids = [s["server"].submit(p, x0, mode=m, precision=s["precision"]) for p, x0, m in s["fits"]]
        got = [s["server"].wait(i) for i in ids]
        return {"x": [r["x"] for r in got], "f": np.array([r["f"] for r in got])}
    ctx = s["ctx"]
    if call == "fit":
        r = B.musr_fit(ctx.ctx, s["x"][0], s["mode"], s["precision"])
        return {"x": r["x"], "f": r["f"]}
    if call == "errors":
        return ctx.gauss_newton(s["x"][0], s["mode"], s["precision"])
    if call == "autograd":
        s["t_x"].grad = None
        f = A.cost(s["t_x"], ctx, s["mode"], s["precision"])
        f.backward()
        return {"value": f.detach(), "grad": s["t_x"].grad}
    if call == "eval_device":
        B.musr_eval_device(ctx.ctx, s["d_x"].data_ptr(), s["d_x"].shape[0], s["mode"], s["precision"], s["grad"], s["d_out"].data_ptr())
        return {"value": s["d_out"][:, 0], "grad": s["d_out"][:, 1:]} if s["grad"] else {"value": s["d_out"][:, 0]}
    if s["x"].shape[0] == 1:
        v, g, _ = ctx.eval(s["x"][0], s["mode"], s["precision"], grad=s["grad"])
    else:
        v, g, _ = ctx.eval_batch(s["x"], s["mode"], s["precision"], grad=s["grad"])
    return {"value": v, "grad": g} if s["grad"] else {"value": v}


def exact(case, seed):
    if case["call"] == "poisson":
        rho, h = _density(case, seed)
        n = rho.shape
        d = [torch.arange(2 * k, dtype=torch.float64, device=DEV) for k in n]
        d = [torch.minimum(v, 2 * k - v) * w for v, k, w in zip(d, n, h)]
        r = (d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2).sqrt()
        r[0, 0, 0] = min(h)
        k = [2 * v for v in n]
        phi = torch.fft.irfftn(torch.fft.rfftn(rho, s=k) * torch.fft.rfftn(1.0 / r), s=k)
        return phi[:n[0], :n[1], :n[2]].clone() * (h[0] * h[1] * h[2])
    if case["call"] == "serve":
        got = [_optimum(p, x0, m) for p, x0, m in _served(case, seed)]
        return {"x": [x for x, _ in got], "f": np.array([float(f) for _, f in got])}
    p = _exact_data(_problem(case["theory"], case["nhist"], case["nbins"], case["dtype"], case["t0"], seed))
    grad = case.get("grad", True)
    x = _vectors(p, case.get("nvec", 1), grad, seed)
    if case["call"] == "fit":
        x, f = _optimum(p, x[0], case["mode"])
        return {"x": x, "f": float(f)}
    if case["call"] == "errors":
        return _gauss_newton(p, x[0], case["mode"])
    got = [_cost(p, v, case["mode"], grad) for v in x]
    value, g = torch.stack([v for v, _ in got]), torch.stack([v for _, v in got])
    if case["call"] == "autograd" or (case["call"] == "eval" and len(got) == 1):
        value, g = (value[0], g[0]) if case["call"] == "autograd" else (float(value[0]), g[0])
    return {"value": value, "grad": g} if grad else {"value": value}


#: Floating operations of one (histogram, bin) pair in the cheapest form of each theory's model (time factors shared by
#: the histograms): cost and gradient, cost alone.
PAIR_FLOPS = {"chi2": (34, 14), "mle": (64, 44)}


def work(case):
    if case["call"] == "poisson":
        n = case["nx"] * case["ny"] * case["nz"]
        # two real transforms of the doubled mesh, of which only the occupied lines need be transformed
        return {"bytes": 16.0 * n, "flops": 2 * 2.5 * 8 * n * math.log2(8 * n) * (1.75 / 3.0)}
    if case["call"] == "serve":
        fits = [(1 if i % 3 == 0 else case["max_hist"] ** 0.5) * (4096 * case["max_bins"]) ** 0.5 for i in range(case["fits"])]
        return {"bytes": 4.0 * sum(fits), "flops": 20 * 49.0 * sum(fits)}
    pairs = case["nhist"] * case["nbins"]
    P = _theory(case["theory"], case["nhist"])[3].size
    size = 8 if case["dtype"] == "fp64" else 4
    if case["theory"] == "asym":
        size = 8  # the asymmetry and its weight
    each = PAIR_FLOPS[case["mode"]][0 if case.get("grad", True) else 1]
    if case["call"] == "fit":  # the curvature's points and about ten steps
        return {"bytes": size * pairs + 16.0 * P, "flops": each * pairs * (P + 10.0)}
    if case["call"] == "errors":
        return {"bytes": size * pairs + 8.0 * P * (P + 1), "flops": each * pairs * 4.0}
    nvec, out = case["nvec"], (1 + P if case.get("grad", True) else 1)
    return {"bytes": size * pairs + 8.0 * nvec * (P + out), "flops": float(each * pairs * nvec)}
