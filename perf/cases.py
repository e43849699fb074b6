"""The calls a user of this package makes, as timed cases.

Three activities make up the use of the library, and every case is one call
(or one request's calls) of them, through ``gp.Context``:

- searching theta: batches of candidates in split precision (the generations
  of the genetic search, the multi-start batches), from the smallest designs
  of the paper's Table 1 to n = 16384;
- refining in double: compass batches and the gradient, one candidate or one
  per start, and the 8 x 8 grid of the small double-precision fit;
- fitting and predicting: the final double fit with its 1000-point SSPE set,
  a serving request (batch, fit of the best, predictions), and kriging at
  1e5 points from a resident model.

Designs are random Latin hypercubes and responses the smooth sums of
``inputs.py``; the double-precision cases keep p <= 1.95 beyond the small
grid (the paper's own choice, for a correlation matrix that is not singular
to working precision).
"""
import math

import numpy as np
import torch

from paper_1203_1269_gb300 import gp, inputs

_DEV = "cuda:0"
_contexts = {}


def _context(corr):
    """One context per correlation family, kept for the life of the process
    (its workspace serves every call, as in a program that fits many data
    sets)."""
    if corr not in _contexts:
        _contexts[corr] = gp.Context(0, correlation=corr)
    return _contexts[corr]


def _case(name, kind, n, d, T, p, delta, prec, N=0, lo=-2.0, corr="powexp"):
    return {"name": name, "kind": kind, "n": n, "d": d, "T": T, "p": p, "delta": delta, "prec": prec,
            "N": N, "lo": lo, "corr": corr}


def listed():
    return [
        # one generation of the genetic search, Table 1's d = 2 designs: launches and latency
        _case("search_n64_d2", "nll", 64, 2, 100, 1.95, 1e-8, "mixed"),
        # one generation at Table 2's third size
        _case("search_n1024_d6", "nll", 1024, 6, 100, 1.95, 1e-8, "mixed"),
        # the benchmark batch: a multi-start population at n = 4000
        _case("search_n4000_d6", "nll", 4000, 6, 256, 1.95, 1e-7, "mixed"),
        # the large instance, a short generation
        _case("search_n16384_d10", "nll", 16384, 10, 8, 1.9, 1e-6, "mixed"),
        # the Matern alternative (nu = 5/2) at the batched study's shape, a ragged n
        _case("matern_n2047_d8", "nll", 2047, 8, 128, 1.95, 1e-6, "mixed", corr="matern52"),
        # the small double-precision fit: the 8 x 8 grid of candidates at n = 200
        _case("grid_n200_d2", "grid", 200, 2, 64, 2.0, 1e-8, "fp64"),
        # one round of the double-precision compass refinement: 2 d neighbours
        _case("compass_n4064_d6", "nll", 4064, 6, 12, 1.95, 1e-7, "fp64", lo=-1.0),
        # one iteration of the multi-start gradient search (16 starts)
        _case("gradient_n1024_d6", "grad", 1024, 6, 16, 1.95, 1e-6, "fp64", lo=-1.0),
        # one step of the gradient refinement of a single candidate
        _case("gradient_n4064_d6", "grad", 4064, 6, 1, 1.95, 1e-6, "fp64", lo=-1.0),
        # the final double fit and the means at its 1000 held-out points (the SSPE's)
        _case("fit_n4064_d6", "fit", 4064, 6, 1, 1.95, 1e-7, "fp64", N=1000, lo=-1.0),
        # a serving request at the middle of its size range: 32 candidates, the
        # fit of the best one, 1000 predictions
        _case("serve_n1448_d7", "serve", 1448, 7, 32, 1.95, 1e-6, "mixed", N=1000),
        # kriging means and variances at 1e5 points from a resident double fit
        _case("krige_n8192_d10", "krige", 8192, 10, 1, 1.9, 1e-6, "fp64", N=100000, lo=-0.5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "double", "grad", "grad", "fit", "serve", "krige"])
    d = rng.randint(2, 12)
    if kind == "search":
        n = _log_int(rng, 16, 12000)
        T = _log_int(rng, 8, min(512, max(8, int(8e12 / n ** 3))) + 1)
        corr = rng.choice(["powexp", "powexp", "powexp", "matern12", "matern32", "matern52"])
        c = _case("", "nll", n, d, T, rng.choice([1.5, 1.9, 1.95, 2.0]), rng.choice([1e-8, 1e-7, 1e-6]), "mixed",
                  corr=corr)
    elif kind == "double":
        n = _log_int(rng, 16, 6000)
        T = _log_int(rng, 1, min(64, max(1, int(3e11 / n ** 3))) + 1)
        c = _case("", "nll", n, d, T, rng.choice([1.5, 1.9, 1.95]), rng.choice([1e-7, 1e-6]), "fp64", lo=-1.0)
    elif kind == "grad":
        n = _log_int(rng, 100, 4500)
        T = _log_int(rng, 1, min(16, max(1, int(1e11 / n ** 3))) + 1)
        c = _case("", "grad", n, d, T, rng.choice([1.5, 1.9, 1.95]), 1e-6, "fp64", lo=-1.0)
    elif kind == "fit":
        c = _case("", "fit", _log_int(rng, 100, 6000), d, 1, rng.choice([1.5, 1.9, 1.95]),
                  rng.choice([1e-7, 1e-6]), "fp64", N=1000, lo=-1.0)
    elif kind == "serve":
        c = _case("", "serve", _log_int(rng, 256, 8192), d, 32, rng.choice([1.5, 1.95, 2.0]),
                  rng.choice([1e-8, 1e-6]), "mixed", N=1000)
    else:
        c = _case("", "krige", _log_int(rng, 500, 8192), rng.randint(8, 12), 1, rng.choice([1.5, 1.9, 1.95]), 1e-6, "fp64",
                  N=_log_int(rng, 1000, 100000), lo=-0.5)
    del c["name"]
    return c


def _data(case, seed):
    """Host arrays of one data set: x, y, the T candidates, N test points."""
    g = inputs.rng(seed)
    n, d = case["n"], case["d"]
    x = inputs.random_lhd(g, n, d)
    y = inputs.y_sinsum(x)
    if case["kind"] == "grid":
        y = inputs.y_trig2(x)
        th = inputs.grid_thetas(2, 8)
    else:
        th = inputs.log_uniform_thetas(g, case["T"], d, lo=case["lo"])
    xs = inputs.uniform_design(g, case["N"], d)
    return x, y, th, xs


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=_DEV)


def prepare(case, seed):
    x, y, th, xs = (_dev(a) for a in _data(case, seed))
    s = dict(case, ctx=_context(case["corr"]), x=x, y=y, th=th, xs=xs)
    if case["kind"] == "krige":
        s["model"] = s["ctx"].fit(x, y, th[0], case["p"], case["delta"], case["prec"])
    return s


def run(s):
    ctx, x, y, th, p, delta, prec = (s[k] for k in ("ctx", "x", "y", "th", "p", "delta", "prec"))
    kind = s["kind"]
    if kind in ("nll", "grid"):
        return ctx.nll_batch(x, y, th, p, delta, prec)
    if kind == "grad":
        return ctx.nll_grad_batch(x, y, th, p, delta)
    if kind == "krige":
        yhat, s2 = ctx.predict(s["model"], s["xs"])
        return {"yhat": yhat, "s2": s2}
    if kind == "fit":
        model = ctx.fit(x, y, th[0], p, delta, prec)
        out = {}
    else:
        out, best, model = ctx.fit_batch(x, y, th, p, delta, prec)
        out = dict(out, best=best)
    out["model"] = [model.nll, model.mu, model.sigma2, model.logdet]
    out["yhat"], s2 = ctx.predict(model, s["xs"], want_var=kind == "serve")
    if kind == "serve":
        out["s2"] = s2
    model.free()
    return out


def work(case):
    """Bytes: the arrays a caller hands over and gets back.  Operations: one
    exponential argument per pair, d multiply-adds each, the n^3 / 3 of every
    factorisation (and 2/3 n^3 more for R^-1 under the gradient), and the n^2
    of a triangular solve per predicted variance."""
    n, d, T, N = case["n"], case["d"], case["T"], case["N"]
    out = {"nll": 4 * T, "grid": 4 * T, "grad": (d + 1) * T, "fit": 4, "serve": 4 * T, "krige": 0}[case["kind"]]
    flops = T * (n ** 3 / 3.0 + 2.0 * d * n * n / 2.0) if case["kind"] != "krige" else 0.0
    if case["kind"] == "grad":
        flops += T * (2.0 / 3.0 * n ** 3 + d * n * n)
    variances = case["kind"] in ("serve", "krige")
    flops += N * (2.0 * d * n + (1.0 * n * n if variances else 0.0))
    held = n * n / 2.0 if case["kind"] == "krige" else 0.0   # the resident factor
    return {"bytes": 8.0 * (n * d + n + T * d + out + N * (d + 1 + variances) + held), "flops": flops}


# ---- the same quantities in plain 64-bit torch -----------------------------

def _powers(a, b, case):
    """|a_k - b_k|^p (or |a_k - b_k| for the Matern families) per dimension."""
    for k in range(case["d"]):
        h = (a[:, k, None] - b[None, :, k]).abs_()
        yield h if case["corr"] != "powexp" else h.pow_(case["p"])


def _corr(powers, theta, case):
    """The correlations of one theta from the per-dimension powers."""
    S, q = 0.0, 1.0
    for k, w in enumerate(powers):
        h = w * theta[k]
        if case["corr"] == "matern32":
            h = h * math.sqrt(3.0)
            q = q * (1.0 + h)
        elif case["corr"] == "matern52":
            h = h * math.sqrt(5.0)
            q = q * (1.0 + h + h * h / 3.0)
        S = S + h
    return torch.exp(-S) * q


def _solve(R, y, delta):
    """L, a = L^-1 1, b = L^-1 y and the scalars of eqs. 3-4 for R + delta I
    (None where R is not positive definite)."""
    n = y.numel()
    R.diagonal().fill_(1.0 + delta)
    L, info = torch.linalg.cholesky_ex(R)
    if int(info) != 0:
        return None
    ab = torch.linalg.solve_triangular(L, torch.stack([torch.ones_like(y), y], 1), upper=False)
    a, b = ab[:, 0], ab[:, 1]
    mu = (a @ b) / (a @ a)
    e = b - mu * a
    Q = e @ e
    logdet = 2.0 * L.diagonal().log().sum()
    return L, a, e, float(logdet + n * torch.log(Q)), float(mu), float(Q / n), float(logdet)


def _exact_predict(L, a, e, mu, sigma2, x, theta, xs, case):
    """Kriging means and variances."""
    w = torch.linalg.solve_triangular(L.T, e[:, None], upper=True)[:, 0]
    z = torch.linalg.solve_triangular(L.T, a[:, None], upper=True)[:, 0]
    aa = a @ a
    yhat, s2 = [], []
    for c in range(0, xs.shape[0], 20000):
        r = _corr(_powers(x, xs[c:c + 20000], case), theta, case)
        yhat.append(mu + r.T @ w)
        v = torch.linalg.solve_triangular(L, r, upper=False)
        u = 1.0 - r.T @ z
        s2.append(sigma2 * (1.0 + case["delta"] - (v * v).sum(0) + u * u / aa))
    return torch.cat(yhat), torch.cat(s2)


def exact(case, seed):
    n, T, kind, delta = case["n"], case["T"], case["kind"], case["delta"]
    x, y, th, xs = (_dev(a) for a in _data(case, seed))
    D = list(_powers(x, x, case))
    nll, mu, s2, ld, grad = [], [], [], [], []
    best = None
    for t in range(T):
        R = _corr(D, th[t], case)
        Rz = R.clone() if kind == "grad" else None
        got = _solve(R, y, delta)
        if got is None:
            for v, bad in ((nll, math.inf), (mu, math.nan), (s2, math.nan), (ld, math.nan)):
                v.append(bad)
            grad.append(torch.full((case["d"],), math.nan, dtype=torch.float64, device=_DEV))
            continue
        L, a, e = got[:3]
        for v, g in zip((nll, mu, s2, ld), got[3:]):
            v.append(g)
        if kind == "grad":
            w = torch.linalg.solve_triangular(L.T, e[:, None], upper=True)[:, 0]
            M = torch.cholesky_inverse(L)
            M.addr_(w, w, alpha=-1.0 / s2[-1])   # (n / Q) w w'
            M.mul_(Rz).fill_diagonal_(0.0)
            grad.append(torch.stack([-(M * Dk).sum() for Dk in D]))
        elif kind in ("fit", "serve", "krige") and (best is None or nll[-1] < nll[best[0]]):
            best = (t, L, a, e)
    col = lambda v: torch.tensor(v, dtype=torch.float64)  # noqa: E731
    if kind == "grad":
        return {"nll": col(nll), "grad": torch.stack(grad), "status": None}
    out = {"nll": col(nll), "mu": col(mu), "sigma2": col(s2), "logdet": col(ld), "status": None}
    if kind in ("nll", "grid"):
        return out
    if best is None:
        return None
    t, L, a, e = best
    yhat, var = _exact_predict(L, a, e, mu[t], s2[t], x, th[t], xs, case)
    if kind == "krige":
        return {"yhat": yhat, "s2": var}
    point = {"model": [nll[t], mu[t], s2[t], ld[t]], "yhat": yhat}
    return point if kind == "fit" else dict(out, best=None, s2=var, **point)
