"""The work a user of this library has it do, as timed cases.

Five kinds of call, all through the public Python entry points:

  run       a whole integration as the paper runs one (Section 3.2): from the uniform grid, an
            adapting warm-up stage, then an adapting production stage; the results, the adapted
            grid and the last iteration's sums are read back.  Optionally with a histogram of the
            integrand's observable, or with VEGAS+ stratification.  The handle is kept between
            calls, as by a program that integrates one process after another.
  gradient  Vegas.adjoint on a warmed-up grid that is held fixed: dsigma/dtheta of Drell-Yan.
  autograd  DrellYanIntegral: sigma(theta) and its backward pass, as inside a fit.
  batch     VegasBatch.iterate: many integrations of uneven size advanced together.

Sizes are those of paper_1503_06182_gb300.workloads, of the benchmark and of the tests.
``exact`` restates the method in 64-bit torch and numpy, without the library.
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_1503_06182_gb300 import vegas as v
from paper_1503_06182_gb300 import workloads as wl
from paper_1503_06182_gb300.autograd import DrellYanIntegral

PARAMS = {"gauss": wl.GAUSS_PARAMS, "dy": wl.DY_PARAMS, "ee3j": wl.EE3J_PARAMS,
          "dy_nlo": wl.DYNLO_PARAMS}
IDS = {"gauss": v.VEGAS_GAUSS, "dy": v.VEGAS_DY, "ee3j": v.VEGAS_EE3J, "dy_nlo": v.VEGAS_DY_NLO}
# drawn dimensions (a narrow peak in more axes than five is found by a handful of a first
# iteration's events, and the grid then follows the last bits of single weights)
MIN_DIM = {"gauss": 2, "dy": 4, "ee3j": 5, "dy_nlo": 5}
MAX_DIM = {"gauss": 5, "dy": 10, "ee3j": 8, "dy_nlo": 13}
# the observable's usual range: x_0, m_ll in GeV, thrust
HIST_RANGE = {"gauss": (0.0, 1.0), "dy": (60.0, 120.0), "ee3j": (0.6, 1.0),
              "dy_nlo": (60.0, 120.0)}
# floating-point operations per event without the grid map (transcendentals and
# divisions as one each) and, for the Gaussian and the NLO factors, per axis
FLOPS = {"gauss": (3, 3), "dy": (94, 0), "ee3j": (130, 0), "dy_nlo": (94, 6)}
GRADIENT_FLOPS = 90  # the reverse sweep's, on top of the Drell-Yan weight's


def _run(name, integrand, ndim, nbins, precision, warm, main, hist=0, strat=False):
    return {"name": name, "kind": "run", "integrand": integrand, "ndim": ndim, "nbins": nbins,
            "precision": precision, "warm_calls": warm[0], "warm_iters": warm[1],
            "calls": main[0], "iters": main[1], "hist": hist, "strat": strat}


def listed():
    return [
        # the paper's own run: 4 x 1,000 warm-up and 10 x 10,000 production events over a
        # 13-dimensional NLO-shaped integral, in the default precision (ten tiles of events)
        _run("paper_nlo13_fp64", "dy_nlo", 13, 50, "fp64", (1000, 4), (10_000, 10)),
        # the same run shape over a 10-dimensional LO integral, FP32 integrand
        _run("paper_lo10_fp32", "dy", 10, 50, "fp32", (1000, 4), (10_000, 10)),
        # a quick default-precision integration of a low-dimensional peak
        _run("gauss4_fp64", "gauss", 4, 50, "fp64", (10_000, 4), (100_000, 5)),
        # the benchmark's workload: a production-quality LO Drell-Yan cross section
        _run("dy_fp32", "dy", 4, 100, "fp32", (100_000, 4), (1_000_000, 10)),
        # the same cross section in the default precision
        _run("dy_fp64", "dy", 4, 100, "fp64", (100_000, 4), (1_000_000, 10)),
        # with the dilepton-mass distribution filled while integrating
        _run("dy_mll60_fp32", "dy", 4, 100, "fp32", (100_000, 4), (1_000_000, 10), hist=60),
        # with adaptive stratified sampling
        _run("dy_plus_fp32", "dy", 4, 100, "fp32", (100_000, 4), (1_000_000, 10), strat=True),
        # an NLO-shaped integral: 13 axes, many transcendentals per event
        _run("nlo13_fp32", "dy_nlo", 13, 50, "fp32", (100_000, 4), (1_000_000, 10)),
        # a high-statistics 3-jet rate, ragged call counts
        _run("ee3j_fp32", "ee3j", 5, 100, "fp32", (1_000_003, 4), (10_000_001, 10)),
        # one step of a fit: cross section and gradient through torch.autograd
        {"name": "fit_step_fp64", "kind": "autograd", "ndim": 4, "nbins": 100,
         "precision": "fp64", "warm_calls": 20_000, "warm_iters": 5, "calls": 100_000,
         "iters": 5},
        # the high-statistics gradient
        {"name": "gradient_fp32", "kind": "gradient", "ndim": 4, "nbins": 100,
         "precision": "fp32", "warm_calls": 100_000, "warm_iters": 4, "calls": 100_000_000,
         "iters": 10},
        # 64 integrations of 2 to 12 axes (the Gaussian's at most 5) and 1e4 to 1e7 calls
        {"name": "batch64_fp32", "kind": "batch", "n": 64, "spec": wl.SEED, "nbins": 100,
         "precision": "fp32", "calls_lo": 10_000, "calls_hi": 10_000_000, "iters": 10},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choices(("run", "autograd", "gradient", "batch"), (12, 2, 2, 1))[0]
    precision = rng.choice(("fp64", "fp32"))
    if kind == "run":
        integrand = rng.choice(("gauss", "dy", "dy", "ee3j", "dy_nlo"))
        ndim = rng.randint(MIN_DIM[integrand], MAX_DIM[integrand])
        nbins = rng.randint(20, 150)
        extra = rng.random()
        strat = extra < 0.15 and integrand in ("gauss", "dy") and ndim <= 6
        if strat:
            precision = "fp32"
        hist = rng.randint(10, 120) if 0.15 <= extra < 0.4 else 0
        hi = 1_000_000 if precision == "fp64" or ndim > 8 else 10_000_000
        calls = _log_int(rng, 10_000, hi)
        iters = rng.randint(3, 10)
        return {"kind": "run", "integrand": integrand, "ndim": ndim, "nbins": nbins,
                "precision": precision, "warm_calls": max(1000, calls // 10),
                "warm_iters": rng.randint(2, 4), "calls": calls, "iters": iters, "hist": hist,
                "strat": strat}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(4, 48), "spec": rng.randrange(1 << 20),
                "nbins": rng.randint(30, 120), "precision": "fp32",
                "calls_lo": _log_int(rng, 5_000, 20_000),
                "calls_hi": _log_int(rng, 100_000, 5_000_000), "iters": rng.randint(4, 10)}
    hi = 1_000_000 if kind == "autograd" or precision == "fp64" else 50_000_000
    calls = _log_int(rng, 20_000, hi)
    return {"kind": kind, "ndim": rng.randint(4, 6), "nbins": rng.randint(40, 120),
            "precision": precision, "warm_calls": 20_000, "warm_iters": rng.randint(3, 5),
            "calls": calls, "iters": rng.randint(3, 10)}


# ------------------------------------------------------------------ the calls
def _members(case):
    spec = wl.batch_spec(case["n"], case["spec"], case["calls_lo"], case["calls_hi"])
    return [replace(m, ndim=min(m.ndim, MAX_DIM["gauss"])) if m.integrand == wl.GAUSS else m
            for m in spec]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        spec = _members(case)
        b = v.VegasBatch([(m.ndim, m.ncall, m.integrand, m.params) for m in spec], case["nbins"],
                         seed, precision=case["precision"])
        return {"case": case, "b": b, "n": len(spec)}
    if kind == "autograd":
        integ = DrellYanIntegral(case["ndim"], case["nbins"], seed, ncall=case["calls"],
                                 itmx=case["iters"], precision=case["precision"])
        integ.warmup(case["warm_calls"], case["warm_iters"])
        theta = [wl.DY_PARAMS[i] for i in wl.DY_GRAD_INDEX]
        theta = torch.tensor(theta, dtype=torch.float64, requires_grad=True)
        return {"case": case, "integ": integ, "theta": theta}
    g = v.Vegas(case["ndim"], case["nbins"], seed, precision=case["precision"])
    if kind == "gradient":
        p = np.array(wl.DY_PARAMS)
        g.iterate(case["warm_calls"], case["warm_iters"], v.VEGAS_DY, p)
        g.set(v.VEGAS_OPT_ADAPT, 0)
        return {"case": case, "g": g, "params": p}
    if case["strat"]:
        g.set(v.VEGAS_OPT_STRAT, 1)
    if case["hist"]:
        g.hist_set(case["hist"], *HIST_RANGE[case["integrand"]])
    uniform = np.tile(np.arange(case["nbins"] + 1) / case["nbins"], (case["ndim"], 1))
    return {"case": case, "g": g, "params": np.array(PARAMS[case["integrand"]]),
            "uniform": uniform}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["b"]
        integral, error, chi2, per = b.iterate(case["iters"])
        grids = np.concatenate([b.grid(i).reshape(-1) for i in range(state["n"])])
        return {"integral": integral, "error": error, "chi2": chi2, "per_iter": per,
                "grid": grids}
    if kind == "autograd":
        sigma = state["integ"](state["theta"])
        grad, = torch.autograd.grad(sigma, state["theta"])
        return {"integral": sigma.detach(), "error": state["integ"].last_error, "grad": grad,
                "grad_err": state["integ"].last_grad_err}
    g = state["g"]
    if kind == "gradient":
        grad, grad_err, integral, error, per = g.adjoint(case["calls"], case["iters"],
                                                         state["params"])
        return {"integral": integral, "error": error, "grad": grad, "grad_err": grad_err,
                "per_iter": per}
    ig, p = IDS[case["integrand"]], state["params"]
    g.grid = state["uniform"]
    g.iterate(case["warm_calls"], case["warm_iters"], ig, p)
    integral, error, chi2, per, _ = g.iterate(case["calls"], case["iters"], ig, p)
    out = {"integral": integral, "error": error, "chi2": chi2, "per_iter": per, "grid": g.grid,
           "last_sums": g.last_sums()}
    if case["hist"]:
        out["hist"], out["hist_err"], _ = g.hist()
    if case["strat"]:
        _, out["counts"], out["variances"] = g.strat()
    return out


def work(case):
    """Per pass: the events' arithmetic; the parameters and the grid in, the results and the grid
    out (the event stream is generated, and the sums stay on the chip)."""
    if case["kind"] == "batch":
        ms = _members(case)
        flops = sum(case["iters"] * m.ncall * _event_flops(("gauss", "dy", "ee3j")[m.integrand],
                                                           m.ndim) for m in ms)
        edges = sum(m.ndim for m in ms) * (case["nbins"] + 1)
        return {"bytes": 8 * (2 * edges + len(ms) * (16 + 2 * case["iters"])), "flops": flops}
    events = case["calls"] * case["iters"]
    edges = case["ndim"] * (case["nbins"] + 1)
    if case["kind"] in ("gradient", "autograd"):
        f = _event_flops("dy", case["ndim"])
        per = f + GRADIENT_FLOPS + (f if case["kind"] == "autograd" else 0)
        return {"bytes": 8 * (edges + 32 + 12 * case["iters"]), "flops": events * per}
    events += case["warm_calls"] * case["warm_iters"]
    return {"bytes": 8 * (3 * edges + 32 + 2 * case["iters"] + 3 * case["hist"]),
            "flops": events * _event_flops(case["integrand"], case["ndim"])}


def _event_flops(integrand, ndim):
    fixed, per_axis = FLOPS[integrand]
    axes = ndim if integrand == "gauss" else max(0, ndim - 4)
    return fixed + per_axis * axes + 5 * ndim


# ------------------------------------------------------------------ in 64 bits
_M32 = 0xFFFFFFFF


def _words(seed, it, batch, first, n, ndim, dev):
    """Philox4x32-10 words of events first..first+n-1: ndim int64 tensors of 32-bit values."""
    ev = torch.arange(first, first + n, dtype=torch.int64, device=dev)
    out = []
    for j in range((ndim + 3) // 4):
        c = [ev & _M32, ev >> 32, torch.full_like(ev, it & _M32),
             torch.full_like(ev, (batch << 8) | j)]
        k0, k1 = seed & _M32, (seed >> 32) & _M32
        for _ in range(10):
            # the 64-bit pattern of each product is exact in wrapping int64 arithmetic
            p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
            c = [((p1 >> 32) & _M32) ^ c[1] ^ k0, p1 & _M32,
                 ((p0 >> 32) & _M32) ^ c[3] ^ k1, p0 & _M32]
            k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
        out += c
    return out[:ndim]


def _sampled(grid, seed, it, batch, first, n):
    """x (list of tensors), bins and the Jacobian of n events on the grid (tensor [d, N+1])."""
    d, N = grid.shape[0], grid.shape[1] - 1
    width = grid[:, 1:] - grid[:, :-1]
    x, bins, J = [], [], 1.0
    for a, r in enumerate(_words(seed, it, batch, first, n, d, grid.device)):
        t = r * N
        i = t >> 32
        f = ((t & _M32).double() + 0.5) * 2.0 ** -32
        w = width[a][i]
        x.append(grid[a][i] + f * w)
        bins.append(i)
        J = J * (w * N)
    return x, bins, J


def _couplings(sw2, kappa):
    """Coefficients of A and B (sums over u, d, s, c, b) of 1, chi_1, chi_2, kappa included."""
    Vl, Al = -0.5 + 2 * sw2, -0.5
    A0 = A1 = A2 = B1 = B2 = 0.0
    for n, Q, T in ((2, 2 / 3, 0.5), (3, -1 / 3, -0.5)):
        Vq, Aq = T - 2 * Q * sw2, T
        A0 += n * Q * Q
        A1 += n * -2 * Q * Vl * Vq * kappa
        A2 += n * (Al * Al + Vl * Vl) * (Aq * Aq + Vq * Vq) * kappa ** 2
        B1 += n * -4 * Q * Al * Aq * kappa
        B2 += n * 8 * Al * Vl * Aq * Vq * kappa ** 2
    return A0, A1, A2, B1, B2


def _drell_yan(x, p, gradient=False):
    """g(x), and dg/d(M_Z, Gamma_Z, sw2, a, b) if asked for."""
    sqrt_s, MZ, GZ, sw2, alpha, mlo, mhi, a, b, norm = p
    s = sqrt_s ** 2
    L, l0 = 2 * math.log(mhi / mlo), math.log(mlo ** 2 / s)
    ltau = l0 + L * x[0]
    ymax = -0.5 * ltau
    y = (2 * x[1] - 1) * ymax
    x1, x2 = torch.exp(y - ymax), torch.exp(-y - ymax)
    u1, u2 = -torch.expm1(y - ymax), -torch.expm1(-y - ymax)  # 1 - x1, 1 - x2
    inside = (u1 > 0) & (u2 > 0)
    u1, u2 = torch.where(inside, u1, 1.0), torch.where(inside, u2, 1.0)
    shat, c = s * x1 * x2, 2 * x[2] - 1
    lu = torch.log(u1 * u2)
    common = 0.2 * norm ** 2 * torch.exp(a * ltau + b * lu)
    lf, lb = common * u2 ** 4, common * u1 ** 4
    sw = lambda z: _couplings(z, 1 / (4 * z * (1 - z)))  # noqa: E731
    A0, A1, A2, B1, B2 = sw(sw2)
    D = shat - MZ ** 2
    den = D ** 2 + (GZ * MZ) ** 2
    r1, r2 = shat * D / den, shat ** 2 / den
    even, odd = (lf + lb) * (1 + c * c), (lf - lb) * c
    P = shat / s * L * 2 * ymax * (alpha ** 2 / 12 * 0.3893794e9 * 4 * math.pi) / shat
    P = torch.where(inside, P, 0.0)
    S = even * (A0 + A1 * r1 + A2 * r2) + odd * (B1 * r1 + B2 * r2)
    if not gradient:
        return P * S
    s1, s2 = even * A1 + odd * B1, even * A2 + odd * B2  # dS/dr1, dS/dr2
    dden = -(s1 * r1 + s2 * r2) / den
    dD = s1 * shat / den + dden * 2 * D
    # derivatives of the coefficients in sw2 by a complex step (exact to rounding)
    _, a1, a2, b1, b2 = (z.imag * 1e30 for z in sw(complex(sw2, 1e-30)))
    return P * S, [P * (dden * 2 * GZ ** 2 * MZ - dD * 2 * MZ), P * dden * 2 * GZ * MZ ** 2,
                   P * (even * (a1 * r1 + a2 * r2) + odd * (b1 * r1 + b2 * r2)),
                   P * S * ltau, P * S * lu]


def _value(integrand, x, p):
    if integrand == "gauss":
        q = sum((t - 0.5) ** 2 for t in x)
        return torch.exp(-q / (2 * p[0] ** 2)) - (p[1] if len(p) > 1 else 0.0)
    if integrand == "dy":
        return _drell_yan(x, p)
    if integrand == "dy_nlo":
        f = _drell_yan(x, p[:10])
        i0 = float(np.i0(p[10]))
        for t in x[4:]:
            f = f * torch.exp(p[10] * torch.cos(2 * math.pi * t)) / i0
        return f
    u1, u2 = 1 - x[0], 1 - x[1]
    inside = (u1 > p[0]) & (u2 > p[0]) & (x[0] + x[1] - 1 > p[0])
    return torch.where(inside, (x[0] ** 2 + x[1] ** 2) / (u1 * u2), 0.0)


def _observable(integrand, x, p):
    if integrand == "gauss":
        return x[0]
    if integrand == "ee3j":
        return torch.maximum(torch.maximum(x[0], x[1]), 2 - x[0] - x[1])
    return p[5] * (p[6] / p[5]) ** x[0]  # m_ll, tau log-uniform


def _refined(edges, d, alpha=1.5):
    """One axis' new edges from its old ones and the bin sums of w^2."""
    N = len(d)
    sm = np.empty(N)
    sm[1:-1] = (d[:-2] + d[1:-1] + d[2:]) / 3
    sm[0], sm[-1] = (d[0] + d[1]) / 2, (d[-2] + d[-1]) / 2
    if not sm.sum() > 0:
        return edges
    rho = sm / sm.sum()
    r = np.zeros(N)
    k = rho > 0
    r[k] = ((1 - rho[k]) / -np.log(rho[k])) ** alpha
    C = np.concatenate([[0.0], np.cumsum(r)])
    target = C[-1] * np.arange(1, N) / N
    lo = np.minimum(np.searchsorted(C[1:], target, side="right"), N - 1)
    new = edges[lo] + (target - C[lo]) * (edges[lo + 1] - edges[lo]) / r[lo]
    return np.concatenate([[0.0], new, [1.0]])


class _Reference:
    """The method in 64 bits, with its own grid and iteration counter."""

    def __init__(self, integrand, params, ndim, nbins, seed, batch=0):
        self.ig, self.p, self.seed, self.batch = integrand, params, seed, batch
        self.grid = np.tile(np.arange(nbins + 1) / nbins, (ndim, 1))
        self.it = 0
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"

    def chunks(self, calls):
        grid = torch.from_numpy(self.grid).to(self.dev)
        for first in range(0, calls, 1 << 21):
            n = min(1 << 21, calls - first)
            yield _sampled(grid, self.seed, self.it, self.batch, first, n)

    @staticmethod
    def mean_sigma(s1, s2, calls):
        m = s1 / calls
        return m, np.sqrt(np.maximum((s2 / calls - m * m) / (calls - 1), 0.0))

    def stage(self, calls, iters, adapt=True, hist=None):
        N = self.grid.shape[1] - 1
        per, hists = [], []
        for _ in range(iters):
            d = np.zeros((len(self.grid), N))
            h = np.zeros((2, hist[0] + 2 if hist else 0))
            s1 = s2 = 0.0
            for x, bins, J in self.chunks(calls):
                w = J * _value(self.ig, x, self.p)
                w2 = w * w
                s1, s2 = s1 + float(w.sum()), s2 + float(w2.sum())
                for a, i in enumerate(bins if adapt else ()):
                    d[a] += torch.bincount(i, weights=w2, minlength=N).cpu().numpy()
                if hist:
                    n, lo, hi = hist
                    t = (_observable(self.ig, x, self.p) - lo) * (n / (hi - lo))
                    b = torch.where(t < 0, 0, 1 + t.clamp(0, n).long())
                    for q, f in enumerate((w, w2)):
                        h[q] += torch.bincount(b, weights=f, minlength=n + 2).cpu().numpy()
            per.append(self.mean_sigma(s1, s2, calls))
            hists.append(self.mean_sigma(h[0], h[1], calls))
            if adapt:
                self.grid = np.stack([_refined(e, q) for e, q in zip(self.grid, d)])
            self.sums = np.concatenate([[s1, s2], d.reshape(-1)])
            self.it += 1
        self.hists = hists
        return np.array(per)

    def gradient(self, calls, iters):
        per, pg = [], []
        for _ in range(iters):
            s = np.zeros((6, 2))
            for x, _, J in self.chunks(calls):
                g, dg = _drell_yan(x, self.p, gradient=True)
                for q, f in enumerate([g] + dg):
                    f = J * f
                    s[q] += float(f.sum()), float((f * f).sum())
            m = [self.mean_sigma(t[0], t[1], calls) for t in s]
            per.append(m[0])
            pg.append(m[1:])
            self.it += 1
        return np.array(per), np.array(pg)


def _combined(per):
    u = 1 / per[:, 1] ** 2
    mean = float((u * per[:, 0]).sum() / u.sum())
    chi2 = float((u * (per[:, 0] - mean) ** 2).sum()) / max(1, len(per) - 1)
    return mean, float(u.sum() ** -0.5), chi2


def _weighted(u, value, sigma):
    """Combination of per-iteration values with the forward weights u."""
    u = u[:, None]
    return ((u * value).sum(0) / u.sum(),
            np.sqrt((u * u * sigma * sigma).sum(0)) / u.sum())


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        outs = []
        for m in _members(case):
            ref = _Reference(("gauss", "dy", "ee3j")[m.integrand], m.params, m.ndim,
                             case["nbins"], seed, m.index)
            per = ref.stage(m.ncall, case["iters"])
            outs.append((*_combined(per), per, ref.grid.reshape(-1)))
        integral, error, chi2, per, grid = zip(*outs)
        return {"integral": np.array(integral), "error": np.array(error), "chi2": np.array(chi2),
                "per_iter": np.array(per), "grid": np.concatenate(grid)}
    if kind in ("autograd", "gradient"):
        ref = _Reference("dy", wl.DY_PARAMS, case["ndim"], case["nbins"], seed)
        ref.stage(case["warm_calls"], case["warm_iters"])
        per, pg = ref.gradient(case["calls"], case["iters"])
        grad, grad_err = _weighted(1 / per[:, 1] ** 2, pg[..., 0], pg[..., 1])
        integral, error, _ = _combined(per)
        out = {"integral": integral, "error": error, "grad": grad, "grad_err": grad_err}
        if kind == "gradient":
            return dict(out, per_iter=pg)
        return dict(out, integral=torch.tensor(integral, dtype=torch.float64),
                    grad=torch.from_numpy(grad))
    if case["strat"]:
        # the next allocation floors a weight of each hypercube: one differing rounding moves
        # events between hypercubes, and a 64-bit run then takes another sample
        return None
    ref = _Reference(case["integrand"], PARAMS[case["integrand"]], case["ndim"], case["nbins"],
                     seed)
    ref.stage(case["warm_calls"], case["warm_iters"])
    hist = (case["hist"], *HIST_RANGE[case["integrand"]]) if case["hist"] else None
    per = ref.stage(case["calls"], case["iters"], hist=hist)
    integral, error, chi2 = _combined(per)
    out = {"integral": integral, "error": error, "chi2": chi2, "per_iter": per,
           "grid": ref.grid, "last_sums": ref.sums}
    if hist:
        h = np.array(ref.hists)
        out["hist"], out["hist_err"] = _weighted(1 / per[:, 1] ** 2, h[:, 0], h[:, 1])
    return out
