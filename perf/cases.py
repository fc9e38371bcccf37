"""Performance cases of the oscillation chain: what users of the library run.

A case names a call of the public Python API (``api.Plan``, ``api.chi2``,
``api.oscprob``, ``api.oscprob_general``) with its sizes and options.  The
inputs (baselines, parameter points, pseudo-data, nuisances) come from the
seed alone; the expected counts behind the pseudo-data and the 64-bit results
of ``exact`` are formed here with plain torch, not with the library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1804_07682_gb300 import api

K_PHASE = 1e3 / (4.0 * 0.1973269804)  # rad MeV / (eV^2 km)
# sin^2 theta12, sin^2 theta13, sin^2 theta23, delta_cp, dm2_21, dm2_32
TRUTH6 = (0.307, 0.0218, 0.545, 1.2 * math.pi, 7.53e-5, 2.44e-3)
SURVIVAL = (0, 1, 4, 5)  # the four parameters of the nue_bar survival chain
FLAVOUR = {"e": 0, "mu": 1, "tau": 2}
TOTAL_EVENTS = 1e5
SIGMA_ETA = 0.02


def listed():
    return [
        # one evaluation of a small reactor fit point inside a minimiser's loop
        # (10^4 nodes, replayed as a graph): launches and latency
        dict(name="point_small", kind="point", prec="ff", chi="pearson", range="juno", nbins=200, nodes=50, nL=1,
             grad=True, spectra=False, graph=True),
        # the full reactor model: eight baselines, 16.4 M nodes, gradient and
        # per-baseline spectra (the benchmark's workload)
        dict(name="point_reactor8", kind="point", prec="ff", chi="poisson", range="reactor", nbins=1000, nodes=16384,
             nL=8, grad=True, spectra=True, graph=False),
        # a line search or a profile from host buffers: chi^2 alone, the phase
        # in double, odd sizes and a baseline count between instantiations
        dict(name="point_host_f64phase", kind="host", prec="f64phase", chi="poisson", range="reactor", nbins=777,
             nodes=1031, nL=3, grad=False),
        # the all-double mode, for reference results and ill-conditioned fits
        dict(name="point_fp64", kind="point", prec="fp64", chi="poisson", range="reactor", nbins=1000, nodes=262,
             nL=8, grad=True, spectra=False, graph=False),
        # a pull-term fit: 4 parameters and 1000 bin nuisances through the
        # autograd Function, forward and backward
        dict(name="nuisance_autograd", kind="autograd", prec="ff", chi="poisson", range="reactor", nbins=1000,
             nodes=4096, nL=8),
        # a delta-chi^2 map: 64 x 64 points, each on a grid of its own order
        dict(name="scan_survival", kind="scan", prec="ff", chi="poisson", channel="", anti=False, npts=4096, nbins=500,
             lo=14.0, hi=18.0, grad=True),
        # the same for nu_mu -> nu_e appearance, six parameters, ragged sizes
        dict(name="scan_appearance", kind="scan", prec="ff", chi="poisson", channel="mu-e", anti=False, npts=1021,
             nbins=333, lo=13.0, hi=17.0, grad=True),
        # nu_mu disappearance at one point with two detectors, with the spectrum
        dict(name="point_disappearance", kind="channel", prec="ff", chi="poisson", channel="mu-mu", anti=True,
             nbins=400, nodes=513, nL=2, grad=True),
        # an ensemble of pseudo-experiments fitted together, 20 iterations each
        dict(name="fits", kind="fit", prec="ff", nsets=2048, nbins=1000, nodes=262, nL=8, iters=20),
        # the bare probability on an energy vector in double
        dict(name="osc_fp64", kind="osc", prec="fp64", channel="", anti=False, n=1000000, nL=1),
        # a few energies only: the call's own cost
        dict(name="osc_few", kind="osc", prec="fp64", channel="", anti=False, n=10000, nL=1),
        # the same for an appearance channel at two detectors, mixed precision,
        # ragged length
        dict(name="osc_appearance_ff", kind="osc", prec="ff", channel="mu-e", anti=False, n=3000017, nL=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, sizes spread over their ranges."""
    kind = rng.choice(["point", "point", "point", "host", "autograd", "scan", "scan", "channel", "fit", "osc", "osc"])
    if kind in ("point", "host", "autograd", "channel"):
        prec = rng.choice(["ff", "ff", "ff", "f64phase", "fp64"])
        top = {"ff": 1.3e8, "f64phase": 2e7, "fp64": 5e6}[prec]
        nL = rng.choice([1, 2, 3, 5, 8] if kind == "channel" else [1, 2, 3, 5, 8, 8, 8, 12])
        nbins = _log_int(rng, 20, 2000)
        nodes = max(3, min(_log_int(rng, 8, 16384), int(top / (nbins * nL))))
        c = dict(kind=kind, prec=prec, chi=rng.choice(["poisson", "pearson"]), nbins=nbins, nodes=nodes, nL=nL)
        if kind == "channel":
            c.update(channel=rng.choice(["mu-e", "mu-mu", "e-tau"]), anti=rng.random() < 0.5, grad=rng.random() < 0.7)
            return c
        c["range"] = rng.choice(["reactor", "juno"])
        if kind == "autograd":
            return c
        c["grad"] = rng.random() < 0.7
        if kind == "point":
            c.update(spectra=rng.random() < 0.4, graph=rng.random() < 0.5)
        return c
    if kind == "scan":
        hi = rng.uniform(12.5, 18.0)
        return dict(kind=kind, prec="ff" if rng.random() < 0.8 else "f64phase", chi="poisson",
                    channel=rng.choice(["", "", "mu-e", "mu-mu"]), anti=rng.random() < 0.5,
                    npts=_log_int(rng, 16, 4096 if hi < 16.5 else 1024), nbins=_log_int(rng, 40, 500),
                    lo=hi - rng.uniform(0.5, 4.0), hi=hi, grad=rng.random() < 0.8)
    if kind == "fit":
        return dict(kind=kind, prec="ff", nsets=_log_int(rng, 64, 2048), nbins=_log_int(rng, 100, 1000),
                    nodes=_log_int(rng, 40, 262), nL=rng.choice([1, 3, 8]), iters=20)
    return dict(kind=kind, prec=rng.choice(["fp64", "fp64", "ff", "f64phase"]), channel=rng.choice(["", "mu-e", "mu-mu"]),
                anti=rng.random() < 0.5, n=_log_int(rng, 10000, 4000000), nL=rng.choice([1, 1, 2, 3]))


# ------------------------------------------------- the model in 64 bits ----
@functools.lru_cache(maxsize=None)
def _gauss_legendre(n):
    """Nodes and weights on [-1, 1] in double: Newton's method on the recurrence."""
    k = np.arange(1, n + 1)
    x = np.cos(math.pi * (k - 0.25) / (n + 0.5))
    for _ in range(100):
        p0, p1 = np.ones(n), x.copy()
        for j in range(1, n):
            p0, p1 = p1, ((2 * j + 1) * x * p1 - j * p0) / (j + 1)
        dp = n * (x * p1 - p0) / ((x - 1) * (x + 1))
        dx = p1 / dp
        x = x - dx
        if np.abs(dx).max() < 1e-15:
            break
    return x[::-1].copy(), (2.0 / ((1 - x) * (1 + x) * dp * dp))[::-1].copy()


def _order(edges, n, L, dm2):
    """The order to integrate with: n, or a smaller one that gives the same
    integrals to rounding (an n-point rule is exact to rounding once n exceeds
    the phase that cos 2x runs through in the bin by a few tens)."""
    half = 0.5 * np.diff(edges)
    turn = 2.0 * K_PHASE * dm2 * np.max(L) * half / edges[:-1] ** 2
    return min(n, int(turn.max() * 1.2) + 32)


def _nodes(edges, n, e_scale):
    x, w = _gauss_legendre(n)
    e = torch.as_tensor(edges, device="cuda")
    x, w = torch.as_tensor(x, device="cuda"), torch.as_tensor(w, device="cuda")
    half, mid = 0.5 * (e[1:] - e[:-1]), 0.5 * (e[1:] + e[:-1])
    E = mid[:, None] + half[:, None] * x
    Es = E * e_scale
    return E, half[:, None] * w * torch.exp(0.87 - 0.16 * Es - 0.091 * Es * Es)


def _coefficients(th, channel, anti):
    """a_ij = -4 Re X_ij, b_ij = 2 Im X_ij for the pairs 21, 31, 32; th [..., 6]."""
    if not channel:
        s12, s13 = th[..., 0], th[..., 1]
        a = torch.stack([-4 * s12 * (1 - s12) * (1 - s13) ** 2, -4 * (1 - s12) * (1 - s13) * s13,
                         -4 * s12 * (1 - s13) * s13], -1)
        return 1.0, a, torch.zeros_like(a)
    s = [torch.sqrt(th[..., q]) for q in range(3)]
    c = [torch.sqrt(1 - th[..., q]) for q in range(3)]
    ep = torch.exp(1j * th[..., 3])
    (s12, s13, s23), (c12, c13, c23) = s, c
    U = [[c12 * c13 + 0j, s12 * c13 + 0j, s13 * ep.conj()],
         [-s12 * c23 - c12 * s23 * s13 * ep, c12 * c23 - s12 * s23 * s13 * ep, s23 * c13 + 0j],
         [s12 * s23 - c12 * c23 * s13 * ep, -c12 * s23 - s12 * c23 * s13 * ep, c23 * c13 + 0j]]
    a, b = (FLAVOUR[f] for f in channel.split("-"))
    X = torch.stack([U[a][i].conj() * U[b][i] * U[a][j] * U[b][j].conj() for i, j in ((1, 0), (2, 0), (2, 1))], -1)
    if anti:
        X = X.conj()
    return float(a == b), -4 * X.real, 2 * X.imag


def _integrals(th, E, W, L, channel, anti):
    """Per-baseline bin integrals [P, nL, nbins]; th [P, 6]."""
    d, a, b = _coefficients(th, channel, anti)
    dm = torch.stack([th[:, 4], th[:, 4] + th[:, 5], th[:, 5]], -1)
    rows = []
    for Lr in L:
        p = torch.full_like(E, d)[None]
        for q in range(3):
            x = (K_PHASE * float(Lr)) * dm[:, q, None, None] / E
            p = p + a[:, q, None, None] * torch.sin(x) ** 2
            if channel:
                p = p + b[:, q, None, None] * torch.sin(2 * x)
        rows.append((W * p).sum(-1))
    return torch.stack(rows, 1)


def _weights(L):
    w = 1.0 / np.asarray(L) ** 2
    return torch.as_tensor(w / w.sum(), device="cuda")


def _chi2_terms(mu, data, chi):
    if chi == "pearson":
        return (data - mu) ** 2 / mu
    return 2 * (mu - data + torch.where(data > 0, data * torch.log(torch.where(data > 0, data, mu) / mu), data))


# ---------------------------------------------------------------- inputs ----
def _inputs(case, seed):
    """Everything that the seed decides: edges, baselines, points, data, nuisances."""
    rng = np.random.default_rng(seed)
    kind, channel = case["kind"], case.get("channel", "")
    beam = kind in ("scan", "channel")
    v = {"e_scale": 1e-3 if beam else 1.0, "channel": channel, "anti": bool(case.get("anti", False))}
    nbins = case["nbins"]
    lo, hi = {"juno": (1.8, 12.0)}.get(case.get("range"), (0.5, 15.0))
    v["edges"] = np.linspace(500.0, 5000.0, nbins + 1) if beam else np.linspace(lo, hi, nbins + 1)
    nL = case.get("nL", 1)
    if beam:
        v["L"] = np.array([810.0, 295.0, 735.0, 700.0, 280.0, 600.0, 550.0, 650.0])[:nL]
    elif case.get("range") == "juno":
        v["L"] = 52.5 + np.concatenate([[0.0], rng.uniform(-1.0, 1.0, nL - 1)])
    else:
        v["L"] = rng.uniform(0.5, 60.0, nL)
    truth = np.array(TRUTH6)
    if kind == "scan":
        npts = case["npts"]
        th = np.repeat(truth[None], npts, 0)
        th[:, 1] = rng.uniform(0.015, 0.03, npts)
        th[:, 5] = rng.uniform(2.3e-3, 2.6e-3, npts)
        v["counts"] = np.maximum(3, np.rint(2.0 ** rng.uniform(case["lo"], case["hi"], npts) / nbins)).astype(np.int64)
    else:
        th = (truth * (1.0 + rng.uniform(-0.05, 0.05, 6)))[None]
    v["theta"] = th
    t = torch.as_tensor(truth, device="cuda")[None]
    n = case["nodes"] if kind != "scan" else int(v["counts"].max())
    E, W = _nodes(v["edges"], _order(v["edges"], n, v["L"], 1.1 * truth[5]), v["e_scale"])
    M = (_weights(v["L"])[None, :, None] * _integrals(t, E, W, v["L"], channel, v["anti"])).sum(1)[0]
    v["norm"] = float(TOTAL_EVENTS / M.sum())
    mu = (v["norm"] * M).cpu().numpy()
    shape = (case["nsets"], nbins) if kind == "fit" else (nbins,)
    v["data"] = rng.poisson(mu, size=shape).astype(np.float64)
    if kind == "autograd":
        v["eta"] = rng.normal(0.0, SIGMA_ETA, nbins)
    return v


def _osc_inputs(case, seed):
    rng = np.random.default_rng(seed)
    beam = bool(case["channel"])
    E = rng.uniform(*((500.0, 5000.0) if beam else (1.8, 12.0)), case["n"])
    L = [810.0, 295.0, 735.0][:case["nL"]] if beam else [52.5, 30.0, 1.7][:case["nL"]]
    return E, L, np.array(TRUTH6) * (1.0 + rng.uniform(-0.05, 0.05, 6))


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x, dtype=np.float64), device="cuda")


def _channel(v):
    return tuple(v["channel"].split("-")) + (v["anti"],) if v["channel"] else None


def prepare(case, seed):
    if case["kind"] == "osc":
        E, L, th = _osc_inputs(case, seed)
        return {"case": case, "E": _dev(E), "L": L, "theta": tuple(th)}
    v = _inputs(case, seed)
    kind = case["kind"]
    npts = case["nsets"] if kind == "fit" else v["theta"].shape[0]
    kw = dict(node_counts=v["counts"]) if kind == "scan" else dict(nodes_per_bin=case["nodes"])
    plan = api.Plan(v["edges"], v["L"], npts=npts, norm=v["norm"], e_scale=v["e_scale"], prec=case["prec"],
                    kind=case.get("chi", "poisson"), max_datasets=npts if kind == "fit" else 0, channel=_channel(v), **kw)
    th = v["theta"] if v["channel"] else v["theta"][:, SURVIVAL]
    s = {"case": case, "plan": plan, "data": _dev(v["data"])}
    if kind == "fit":
        s["start"] = _dev(np.repeat(th, npts, 0))
    elif kind == "host":
        s["theta"], s["data"] = np.ascontiguousarray(th), v["data"]
    elif kind == "autograd":
        s["theta"], s["eta"] = _dev(th[0]).requires_grad_(), _dev(v["eta"]).requires_grad_()
    else:
        s["theta"] = plan.params_tensor(th)
    if case.get("graph") or (kind == "scan" and not v["channel"]):
        # replayed as a graph: the outputs stay at the same place
        plan.set_graph(True)
        out = {"chi2": torch.empty(npts, dtype=torch.float64, device="cuda")}
        if case["grad"]:
            out["grad"] = torch.empty(npts, 4, dtype=torch.float64, device="cuda")
        if case.get("spectra"):
            out["spectra"] = torch.empty(npts, len(v["L"]), case["nbins"], dtype=torch.float64, device="cuda")
        s["out"] = out
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "osc":
        if case["channel"]:
            a, b = case["channel"].split("-")
            return api.oscprob_general(s["E"], s["L"], s["theta"], a, b, anti=bool(case["anti"]), prec=case["prec"])
        return api.oscprob(s["E"], s["L"], [s["theta"][q] for q in SURVIVAL], case["prec"])
    plan = s["plan"]
    if kind == "point" or (kind == "scan" and not case["channel"]):
        return plan.eval(s["theta"], s["data"], grad=case["grad"], spectra=bool(case.get("spectra")), out=s.get("out"))
    if kind in ("scan", "channel"):
        return plan.eval_general(s["theta"], s["data"], grad=case["grad"], mu=kind == "channel")
    if kind == "host":
        c, g = plan.eval_host(s["theta"], s["data"], grad=case["grad"])
        return {"chi2": c, "grad": g} if case["grad"] else {"chi2": c}
    if kind == "autograd":
        s["theta"].grad = s["eta"].grad = None
        chi2 = api.chi2(s["theta"], plan, s["data"], s["eta"], SIGMA_ETA)
        chi2.backward()
        return {"chi2": chi2.detach(), "grad": s["theta"].grad, "grad_eta": s["eta"].grad}
    params, chi2 = plan.fit(s["start"].clone(), s["data"], iters=case["iters"])
    return {"chi2": chi2, "s2_12": params[:, 0], "s2_13": params[:, 1], "dm2_21": params[:, 2], "dm2_32": params[:, 3]}


# ------------------------------------------------------- work, tolerance ----
def _counts(case):
    """(probabilities evaluated, energy nodes read) of one pass; points of equal
    order share a grid, which is then read once."""
    if case["kind"] == "osc":
        return case["n"] * case["nL"], case["n"]
    if case["kind"] == "scan":
        # the mean of 2^U(lo, hi) nodes a point
        n = case["npts"] * (2.0 ** case["hi"] - 2.0 ** case["lo"]) / ((case["hi"] - case["lo"]) * math.log(2.0))
        orders = [2.0 ** case[k] / case["nbins"] for k in ("lo", "hi")]
        return n, min(n, case["nbins"] * (orders[1] ** 2 - orders[0] ** 2) / 2)
    nodes = case["nbins"] * case["nodes"]
    times = case["nsets"] * case["iters"] if case["kind"] == "fit" else 1
    return nodes * case["nL"] * times, nodes


def work(case):
    """A probability takes two phases reduced modulo pi (8 operations each),
    their sines and cosines (10 each: 20), the third pair by angle addition and
    three products (8), 44 in all; its gradient 10 more.  A node is read as
    1/E and its weight in double (16 bytes)."""
    p, n = _counts(case)
    grad = case["kind"] in ("autograd", "fit") or case.get("grad", False)
    size = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "osc":
        return {"bytes": 8.0 * n + size * p, "flops": 44.0 * p}
    npts = case.get("nsets", case.get("npts", 1))
    values = npts * (case["nbins"] if case["kind"] == "fit" else 8) + 2 * case["nbins"]
    if case.get("spectra"):
        values += case["nL"] * case["nbins"]
    return {"bytes": 16.0 * n + 8.0 * values, "flops": (54.0 if grad else 44.0) * p}


def tolerance(case):
    """About four times the largest difference from ``exact`` seen over the
    listed cases and fifty drawn ones."""
    kind, fp64 = case["kind"], case["prec"] == "fp64"
    if kind == "osc":
        # phases of up to a few hundred rad carry 2^-53 of themselves in
        # double (seen 7e-16), 6e-8 rad in the mixed precisions (seen 3e-7,
        # relative to an appearance probability)
        return {"rel": 1e-14, "max": 1e-13} if fp64 else {"rel": 1.2e-6, "max": 2e-5}
    if kind == "fit":
        # the parameters end where chi^2 no longer falls beyond its rounding
        # (seen 1.3e-5 of a parameter)
        return {"rel": 1e-4, "max": 1e-3}
    if fp64:
        # quadrature weights of order n carry up to n roundings (seen 2e-14)
        return {"rel": 1e-12, "max": 1e-11}
    if case.get("grad", False) or kind == "autograd":
        # near a minimum the gradient is a small difference of the bins'
        # terms, each good to 1e-7 (seen 1.2e-4 of its norm)
        return {"rel": 5e-4, "max": 5e-3}
    return {"rel": 4e-6, "max": 4e-5}  # chi^2 alone (seen 8e-7)


# ----------------------------------------------------------------- exact ----
def exact(case, seed):
    if case["kind"] == "osc":
        E, L, th = _osc_inputs(case, seed)
        E, t = _dev(E), torch.as_tensor(th, device="cuda")[None]
        d, a, b = _coefficients(t, case["channel"], bool(case["anti"]))
        dm = (th[4], th[4] + th[5], th[5])
        out = torch.full((len(L), E.numel()), d, dtype=torch.float64, device="cuda")
        for r, Lr in enumerate(L):
            for q in range(3):
                x = K_PHASE * Lr * dm[q] / E
                out[r] += a[0, q] * torch.sin(x) ** 2 + b[0, q] * torch.sin(2 * x)
        return out
    v = _inputs(case, seed)
    om, channel = _weights(v["L"]), v["channel"]
    if case["kind"] == "fit":
        return _exact_fit(case, v, om)
    par = list(range(6)) if channel else list(SURVIVAL)
    data = _dev(v["data"])
    eta = _dev(v["eta"]).requires_grad_() if "eta" in v else None
    npts = v["theta"].shape[0]
    n_all = v["counts"] if case["kind"] == "scan" else np.full(npts, case["nodes"])
    n_eff = np.array([_order(v["edges"], int(n), v["L"], 1.1 * TRUTH6[5]) for n in n_all])
    chi2 = torch.empty(npts, dtype=torch.float64, device="cuda")
    grad = torch.empty(npts, len(par), dtype=torch.float64, device="cuda")
    for n in np.unique(n_eff):
        E, W = _nodes(v["edges"], int(n), v["e_scale"])
        which = np.flatnonzero(n_eff == n)
        step = max(1, int(2e7 / (E.numel() * len(v["L"]))))
        for k in range(0, which.size, step):
            at = torch.as_tensor(which[k:k + step], device="cuda")
            th = torch.as_tensor(v["theta"][which[k:k + step]], device="cuda").requires_grad_()
            mu_r = _integrals(th, E, W, v["L"], channel, v["anti"])
            mu = v["norm"] * (om[None, :, None] * mu_r).sum(1)
            if eta is not None:
                mu = mu * (1 + eta)
            c = _chi2_terms(mu, data, case["chi"]).sum(-1)
            if eta is not None:
                c = c + ((eta / SIGMA_ETA) ** 2).sum()
            c.sum().backward()
            chi2[at] = c.detach()
            grad[at] = th.grad[:, par]
    if case["kind"] == "autograd":
        return {"chi2": chi2[0], "grad": grad[0], "grad_eta": eta.grad}
    out = {"chi2": chi2}
    if case["grad"]:
        out["grad"] = grad
    if case.get("spectra"):
        out["spectra"] = mu_r.detach()
    if case["kind"] == "channel":
        out["mu"] = mu.detach()
    return out


def _exact_fit(case, v, om):
    """The batched Levenberg-Marquardt fits of ``Plan.fit`` in 64 bits: one
    evaluation an iteration, accepted (damping / 10) if chi^2 fell, else
    rejected (x 10), then (H + lam diag H) delta = -g from the best point,
    H = J^T (2 / mu) J, clamped into the parameters' box."""
    E, W = _nodes(v["edges"], _order(v["edges"], case["nodes"], v["L"], 1.3 * TRUTH6[5]), 1.0)
    data = _dev(v["data"])
    n, nbins = data.shape
    th = _dev(np.repeat(v["theta"][:, SURVIVAL], n, 0))
    best, c_best, lam = th.clone(), torch.full((n,), math.inf, dtype=th.dtype, device="cuda"), torch.full(
        (n,), 1e-3, dtype=th.dtype, device="cuda")
    g_best, H_best = torch.zeros_like(th), torch.zeros(n, 4, 4, dtype=th.dtype, device="cuda")
    lo = torch.tensor([1e-6, 1e-6, 1e-7, 1e-7], dtype=th.dtype, device="cuda")
    hi = torch.tensor([1 - 1e-6, 1 - 1e-6, math.inf, math.inf], dtype=th.dtype, device="cuda")
    step = max(1, int(2e7 / E.numel()))
    for _ in range(case["iters"]):
        M = torch.zeros(n, nbins, dtype=th.dtype, device="cuda")
        J = torch.zeros(n, 4, nbins, dtype=th.dtype, device="cuda")
        for k in range(0, n, step):
            sl = slice(k, k + step)
            s12, s13, d21, d32 = (th[sl, q, None] for q in range(4))
            A = (4 * s12 * (1 - s12) * (1 - s13) ** 2, 4 * (1 - s12) * (1 - s13) * s13, 4 * s12 * (1 - s13) * s13)
            A12 = (4 * (1 - 2 * s12) * (1 - s13) ** 2, -4 * (1 - s13) * s13, 4 * (1 - s13) * s13)
            A13 = (-8 * s12 * (1 - s12) * (1 - s13), 4 * (1 - s12) * (1 - 2 * s13), 4 * s12 * (1 - 2 * s13))
            for w, Lr in zip(om, v["L"]):
                kl = K_PHASE * float(Lr) / E
                M[sl] += w * W.sum(-1)
                for q, dm in enumerate((d21, d21 + d32, d32)):
                    x = dm[..., None] * kl
                    S = w * (W * torch.sin(x) ** 2).sum(-1)
                    D = w * (W * kl * torch.sin(2 * x)).sum(-1)
                    M[sl] -= A[q] * S
                    J[sl, 0] -= A12[q] * S
                    J[sl, 1] -= A13[q] * S
                    if q != 2:
                        J[sl, 2] -= A[q] * D
                    if q != 0:
                        J[sl, 3] -= A[q] * D
        mu, J = v["norm"] * M, v["norm"] * J
        c = _chi2_terms(mu, data, "poisson").sum(-1)
        g = (2 * (1 - data / mu)[:, None] * J).sum(-1)
        H = torch.einsum("pin,pjn->pij", J * (2 / mu)[:, None], J)
        ok = c < c_best
        c_best = torch.where(ok, c, c_best)
        best = torch.where(ok[:, None], th, best)
        g_best = torch.where(ok[:, None], g, g_best)
        H_best = torch.where(ok[:, None, None], H, H_best)
        lam = torch.where(ok, lam / 10, lam * 10)
        # scaled to a unit diagonal for the solve
        d = torch.sqrt(torch.diagonal(H_best, dim1=1, dim2=2))
        Hs = H_best / (d[:, :, None] * d[:, None, :]) + torch.diag_embed(lam[:, None].expand(n, 4))
        th = torch.clamp(best + torch.linalg.solve(Hs, -(g_best / d)[..., None])[..., 0] / d, lo, hi)
    return {"chi2": c_best, "s2_12": best[:, 0], "s2_13": best[:, 1], "dm2_21": best[:, 2], "dm2_32": best[:, 3]}
