"""Performance cases of the library: what its users have it do, and how big.

Every case goes through one public entry point of the package (one step of the
method, or the whole method on one series or on many).  Series are drawn on
the GPU from a seed: a random acyclic instantaneous graph, non-Gaussian shocks
and, where the step under measure fits a VAR, lagged effects.  `exact` restates
each step in plain float64 torch, sharing no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2409_05500_gb300 as vl

NOISES = ("uniform", "laplace", "t3", "powgauss")
PRECISIONS = ("mixed", "mixed_certified", "fp64")
_handles = {}


def _handle() -> "vl.Handle":
    """A program keeps one handle for all the series it fits."""
    dev = torch.cuda.current_device()
    if dev not in _handles:
        _handles[dev] = vl.Handle(dev)
    return _handles[dev]


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # whole method, smallest call: a handful of sensors, where launches count
        {"name": "fit-small", "op": "fit", "prec": "mixed", "m": 10, "n": 1000, "p": 1,
         "noise": "uniform"},
        # whole method, the benchmark's workload: a stock index's daily returns
        {"name": "fit-finance", "op": "fit", "prec": "mixed", "m": 400, "n": 2500, "p": 1,
         "noise": "t3"},
        # whole method with every near tie decided to FP64 accuracy: server monitoring,
        # a long series with three lags
        {"name": "fit-certified-server", "op": "fit", "prec": "mixed_certified", "m": 120,
         "n": 10000, "p": 3, "noise": "laplace"},
        # VAR fit alone with several lags, odd sizes from the middle of the batch's range:
        # the normal equations have 609 rows
        {"name": "var_fit-lags", "op": "var_fit", "prec": "mixed", "m": 203, "n": 4001, "p": 3,
         "noise": "laplace"},
        # pairwise measure of brain regions: few samples, odd count
        {"name": "measure-fmri", "op": "measure", "prec": "mixed", "m": 50, "n": 199,
         "noise": "powgauss"},
        # pairwise measure at the size sweep's top: the largest single call
        {"name": "measure-stretch", "op": "measure", "prec": "mixed", "m": 1600, "n": 4999,
         "noise": "t3"},
        # pairwise measure in plain FP64, for a program that wants no FP32 anywhere
        {"name": "measure-fp64", "op": "measure", "prec": "fp64", "m": 120, "n": 9997,
         "noise": "laplace"},
        # the ordering on a precomputed measure, with its gaps: the size sweep's middle
        {"name": "order-stretch", "op": "order", "m": 800, "noise": "t3"},
        # B0 and B_tau along a known order (a domain's causal order, or a pruned refit)
        {"name": "fit_b-finance", "op": "fit_b", "prec": "mixed", "m": 400, "n": 2499, "p": 1,
         "noise": "t3"},
        # many series of uneven sizes in one call
        {"name": "batched-mixed-sizes", "op": "batched", "prec": "mixed", "count": 48,
         "m_lo": 20, "m_hi": 400, "n_lo": 250, "n_hi": 5000},
        # edge probabilities over moving-block resamples of one series
        {"name": "bootstrap", "op": "bootstrap", "prec": "mixed_certified", "m": 100, "n": 1000,
         "p": 1, "resamples": 64, "block": 50, "noise": "uniform"},
        # the iterative search that the ordering approximates
        {"name": "standard-search", "op": "standard", "prec": "mixed", "m": 100, "n": 999,
         "noise": "uniform"},
    ]


def _logint(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("fit", "fit", "var_fit", "measure", "measure", "order", "fit_b", "batched",
                     "bootstrap", "standard"))
    noise = rng.choice(NOISES)
    if op == "fit":
        prec = rng.choice(("mixed", "mixed", "mixed_certified", "fp64"))
        while True:
            m, n, p = _logint(rng, 10, 400), _logint(rng, 200, 10000), rng.randint(1, 3)
            # enough samples per coefficient for the fit to mean something
            if n - p >= 2 * (m * p + 1) and (prec != "fp64" or m * m * n <= 60 * 60 * 10000):
                break
        return {"op": op, "prec": prec, "m": m, "n": n, "p": p, "noise": noise}
    if op == "var_fit":
        prec = rng.choice(("mixed", "mixed", "fp64"))
        while True:
            m, n, p = _logint(rng, 10, 400), _logint(rng, 200, 10000), rng.randint(1, 3)
            if n - p >= 2 * (m * p + 1) and (prec != "fp64" or (m * p) ** 2 * n <= 3e8):
                break
        return {"op": op, "prec": prec, "m": m, "n": n, "p": p, "noise": noise}
    if op == "measure":
        prec = rng.choice(("mixed", "mixed", "fp64"))
        cap = 120 * 120 * 9997 if prec == "fp64" else 1600 * 1600 * 4999
        while True:
            m, n = _logint(rng, 10, 1600), _logint(rng, 100, 10000)
            if m * m * n <= cap:
                break
        return {"op": op, "prec": prec, "m": m, "n": n, "noise": noise}
    if op == "order":
        return {"op": op, "m": _logint(rng, 10, 1600), "noise": noise}
    if op == "fit_b":
        prec = rng.choice(("mixed", "mixed", "fp64"))
        while True:
            m, n, p = _logint(rng, 10, 800), _logint(rng, 200, 5000), rng.randint(0, 3)
            if n >= 2 * m and (prec != "fp64" or m <= 200):
                break
        return {"op": op, "prec": prec, "m": m, "n": n, "p": p, "noise": noise}
    if op == "batched":
        return {"op": op, "prec": rng.choice(("mixed", "mixed_certified")),
                "count": rng.randint(8, 48), "m_lo": 20, "m_hi": rng.randint(60, 400),
                "n_lo": 250, "n_hi": rng.randint(1000, 5000)}
    if op == "bootstrap":
        n = _logint(rng, 250, 1000)
        return {"op": op, "prec": rng.choice(("mixed", "mixed_certified")),
                "m": _logint(rng, 10, 100), "n": n, "p": 1, "resamples": rng.randint(16, 64),
                "block": rng.randint(10, n // 5), "noise": noise}
    return {"op": "standard", "prec": "mixed", "m": _logint(rng, 10, 100),
            "n": _logint(rng, 200, 1000), "noise": noise}


# ----------------------------------------------------------------- the data
def _shocks(g, kind, m, n):
    """Unit-variance shocks of the named family, m x n."""
    dev = g.device

    def normal():
        return torch.randn((m, n), generator=g, device=dev, dtype=torch.float64)

    if kind == "uniform":
        u = torch.rand((m, n), generator=g, device=dev, dtype=torch.float64)
        return (u - 0.5) * math.sqrt(12.0)
    if kind == "laplace":
        u = torch.rand((m, n), generator=g, device=dev, dtype=torch.float64) - 0.5
        return -torch.sign(u) * torch.log1p(-2.0 * u.abs()) / math.sqrt(2.0)
    if kind == "t3":
        z = normal()
        c = normal() ** 2 + normal() ** 2 + normal() ** 2
        return z / torch.sqrt(c)
    z = normal()
    return torch.sign(z) * z.abs() ** 1.5 / math.sqrt(2.0 * math.sqrt(2.0 / math.pi))


def _mixed(g, noise, m, n):
    """Shocks through a random acyclic graph (about 2.7 parents per variable):
    the residuals of a VAR, m x n, and the order of causes."""
    dev = g.device
    f64 = dict(device=dev, dtype=torch.float64)
    perm = torch.randperm(m, generator=g, device=dev)
    keep = torch.rand((m, m), generator=g, **f64) < min(0.3, 2.7 / max(m - 1, 1))
    w = 0.1 + 0.4 * torch.rand((m, m), generator=g, **f64)
    sgn = torch.where(torch.rand((m, m), generator=g, **f64) < 0.5, -1.0, 1.0)
    L = torch.tril(w * sgn * keep, -1)
    e = _shocks(g, noise, m, n)
    # x = L x + e in causal coordinates
    x = torch.linalg.solve_triangular(torch.eye(m, **f64) - L, e, upper=False, unitriangular=True)
    out = torch.empty((m, n), **f64)  # the solve leaves columns contiguous
    out[perm] = x
    return out, perm.to(torch.int32)


def _lagged(g, m, p):
    """Lagged effects M (p x m x m), spectral radius about 0.5."""
    M = torch.randn((p, m, m), generator=g, device=g.device, dtype=torch.float64)
    for tau in range(p):
        M[tau] *= 0.5 ** (tau + 1) / math.sqrt(m * p)
    return M


def _series(g, noise, m, n, p):
    """A series x_t = sum_tau M_tau x_{t-tau} + shocks, m x n: the recursion
    unrolled to a depth at which the lagged effects have died out."""
    burn, depth = 64, 16
    s, _ = _mixed(g, noise, m, n + burn)
    M = _lagged(g, m, p)
    x = s
    for _ in range(depth):
        y = s.clone()
        for tau in range(1, p + 1):
            y[:, tau:] += M[tau - 1] @ x[:, :-tau]
        x = y
    return x[:, burn:].contiguous()


def _shapes(case, seed):
    """Sizes of the series of a batch: the sizes are the case's own, whatever the seed."""
    rng = np.random.RandomState(case["count"] * 7919 + case["m_hi"] * 31 + case["n_hi"])
    out = []
    for k in range(case["count"]):
        while True:
            m = int(rng.randint(case["m_lo"], case["m_hi"] + 1))
            n = int(rng.randint(case["n_lo"], case["n_hi"] + 1))
            p = int(rng.randint(1, 4))
            if n - p >= 2 * (m * p + 1):
                break
        out.append((m, n, p, NOISES[int(rng.randint(0, 3))]))
    return out


def _inputs(case, seed):
    g = torch.Generator(device=torch.device("cuda", torch.cuda.current_device()))
    g.manual_seed(int(seed) * 1000003 + 17)
    op = case["op"]
    if op in ("fit", "var_fit", "bootstrap"):
        return {"X": _series(g, case["noise"], case["m"], case["n"], case["p"])}
    if op in ("measure", "standard"):
        return {"E": _mixed(g, case["noise"], case["m"], case["n"])[0]}
    if op == "order":
        E, _ = _mixed(g, case["noise"], case["m"], 500)
        return {"D": _measure(E, torch.float32)[2].contiguous()}
    if op == "fit_b":
        E, order = _mixed(g, case["noise"], case["m"], case["n"])
        p = case["p"]
        return {"E": E, "order": order, "M": _lagged(g, case["m"], p) if p else None}
    return {"X": [_series(g, noise, m, n, p) for m, n, p, noise in _shapes(case, seed)]}


def prepare(case, seed):
    st = dict(case, h=_handle(), **_inputs(case, seed))
    dev = torch.device("cuda", torch.cuda.current_device())
    f64 = dict(dtype=torch.float64, device=dev)
    i32 = dict(dtype=torch.int32, device=dev)
    op = case["op"]
    if op == "fit":
        st["out"] = vl.alloc_outputs(case["m"], case["p"])
    elif op == "var_fit":
        m, n, p = case["m"], case["n"], case["p"]
        st["out"] = {"M": torch.empty((p, m, m), **f64), "E": torch.empty((m, n - p), **f64)}
    elif op == "measure":
        m = case["m"]
        st["out"] = {"Hx": torch.empty(m, **f64), "Hr": torch.empty((m, m), **f64),
                     "D": torch.empty((m, m), **f64)}
    elif op in ("order", "standard"):
        st["out"] = {"order": torch.empty(case["m"], **i32), "gap": torch.empty(case["m"], **f64)}
    elif op == "fit_b":
        m, p = case["m"], case["p"]
        st["out"] = {"B0": torch.empty((m, m), **f64)}
        if p:
            st["out"]["Btau"] = torch.empty((p, m, m), **f64)
    elif op == "bootstrap":
        m = case["m"]
        st["out"] = {"edge_prob": torch.empty((m, m), **f64),
                     "order_prob": torch.empty((m, m), **f64)}
    else:  # a batch: one buffer per kind of output, a view of it per series
        shapes = _shapes(case, seed)
        sizes = {"order": [m for m, _, _, _ in shapes], "B0": [m * m for m, _, _, _ in shapes],
                 "M": [p * m * m for m, _, p, _ in shapes]}
        sizes["Btau"] = sizes["M"]
        st["out"] = {k: torch.empty(sum(v), **(i32 if k == "order" else f64))
                     for k, v in sizes.items()}
        parts = {k: torch.split(st["out"][k], sizes[k]) for k in sizes}
        st["instances"] = [
            {"X": X, "p": p, "order": parts["order"][k], "B0": parts["B0"][k].view(m, m),
             "M": parts["M"][k].view(p, m, m), "Btau": parts["Btau"][k].view(p, m, m)}
            for k, (X, (m, _, p, _)) in enumerate(zip(st["X"], shapes))]
    return st


def run(st):
    op, h, o = st["op"], st["h"], st["out"]
    if op == "fit":
        vl.vl_fit(h, st["X"], st["p"], st["prec"], o["M"], o["order"], o["B0"], o["Btau"], o["D"])
    elif op == "var_fit":
        vl.vl_var_fit(h, st["X"], st["p"], st["prec"], o["M"], o["E"])
    elif op == "measure":
        vl.vl_pairwise_measure(h, st["E"], st["prec"], o["Hx"], o["Hr"], o["D"])
    elif op == "order":
        vl.vl_causal_order(h, st["D"], o["order"], o["gap"])
    elif op == "fit_b":
        vl.vl_fit_b(h, st["E"], st["order"], st["M"], st["prec"], o["B0"], o.get("Btau"))
    elif op == "batched":
        status = vl.vl_fit_batched(h, st["instances"], st["prec"])
        return dict(o, status=np.asarray(status, dtype=np.int32))
    elif op == "bootstrap":
        vl.vl_bootstrap(h, st["X"], st["p"], st["resamples"], st["block"], 1, 0.05, st["prec"],
                        o["edge_prob"], o["order_prob"])
    else:
        vl.vl_causal_order_standard(h, st["E"], st["prec"], o["order"], o["gap"])
    return o


# ------------------------------------------------------- least work of a pass
# Operations of one residual sample of the measure: the residual and its scale,
# |u|, two exponentials and a logarithm with their arguments, two sums.
_OPS = 14


def _work_fit(m, n, p):
    ne, mp = n - p, m * p
    b = 8 * (m * n + 2 * p * m * m + 2 * m * m) + 4 * m
    f = ne * m * (mp + m) * 2 + mp ** 3 / 3 + 2 * mp * mp * m + 2 * m * mp * ne  # VAR
    f += ne * m * m + m * (m - 1) * ne * _OPS                                    # measure
    f += 2 * m * m + m ** 3 / 3 + m ** 3 / 3 + 2 * p * m ** 3                    # order, B
    return b, f


def work(case):
    op = case["op"]
    if op == "fit":
        b, f = _work_fit(case["m"], case["n"], case["p"])
    elif op == "var_fit":
        m, n, p = case["m"], case["n"], case["p"]
        ne, mp = n - p, m * p
        b = 8 * (m * n + p * m * m + m * ne)
        f = ne * m * (mp + m) * 2 + mp ** 3 / 3 + 2 * mp * mp * m + 2 * m * mp * ne
    elif op == "measure":
        m, n = case["m"], case["n"]
        b, f = 8 * (m * n + 2 * m * m + m), n * m * m + m * (m - 1) * n * _OPS
    elif op == "order":
        m = case["m"]
        b, f = 8 * m * m + 12 * m, 4 * m * m
    elif op == "fit_b":
        m, n, p = case["m"], case["n"], case["p"]
        b = 8 * (m * n + m * m + 2 * p * m * m) + 4 * m
        f = n * m * m + 2 * m ** 3 / 3 + 2 * p * m ** 3
    elif op == "batched":
        each = [_work_fit(m, n, p) for m, n, p, _ in _shapes(case, 0)]
        b, f = sum(x for x, _ in each), sum(x for _, x in each)
    elif op == "bootstrap":
        m = case["m"]
        _, f = _work_fit(m, case["n"], case["p"])
        b, f = 8 * (m * case["n"] + 2 * m * m), case["resamples"] * f
    else:
        m, n = case["m"], case["n"]
        b = 8 * (m * n + m) + 4 * m
        f = sum(u * (u - 1) * n * _OPS + n * u * u + 2 * u * n for u in range(2, m + 1))
    return {"bytes": float(b), "flops": float(f)}


# ------------------------------------------------------------ 64-bit restatement
def _var(X, p):
    """Least squares of the VAR with intercept: M (p x m x m), E (m x (n - p))."""
    m, n = X.shape
    Y = X[:, p:]
    Z = torch.cat([X[:, p - tau:n - tau] for tau in range(1, p + 1)])
    Yc, Zc = Y - Y.mean(1, keepdim=True), Z - Z.mean(1, keepdim=True)
    Q, R = torch.linalg.qr(Zc.T)
    beta = torch.linalg.solve_triangular(R, Q.T @ Yc.T, upper=True)  # mp x m
    E = Yc - beta.T @ Zc
    M = torch.stack([beta[tau * m:(tau + 1) * m].T for tau in range(p)])
    return M, E


def _entropy(u):
    """Maximum-entropy approximation of the entropy of standardized u (last axis)."""
    a = u.abs()
    A = (a + torch.log1p(torch.exp(-2.0 * a)) - math.log(2.0)).mean(-1, dtype=torch.float64)
    B = (u * torch.exp(-0.5 * u * u)).mean(-1, dtype=torch.float64)
    return 0.5 * (1 + math.log(2 * math.pi)) - 79.047 * (A - 0.37457) ** 2 - 7.4129 * B ** 2


def _measure(E, dtype=torch.float64):
    """Hx, Hr (H of the residual of i on j) and D; the functions in `dtype`."""
    m, n = E.shape
    x = E - E.mean(1, keepdim=True)
    x = x / torch.sqrt((x * x).mean(1, keepdim=True))
    rho = x @ x.T / n
    Hx = _entropy(x.to(dtype))
    xs = x.to(dtype)
    Hr = torch.zeros((m, m), dtype=torch.float64, device=E.device)
    rows = max(1, int(3e7 // (m * n)))
    for i in range(0, m, rows):
        r = rho[i:i + rows].to(dtype)
        sc = 1.0 / torch.sqrt(torch.clamp(1.0 - r * r, min=1e-12))
        Hr[i:i + rows] = _entropy((xs[i:i + rows, None, :] - r[:, :, None] * xs[None]) * sc[:, :, None])
    Hr.fill_diagonal_(0.0)
    D = Hx[None, :] + Hr - Hx[:, None] - Hr.T
    D.fill_diagonal_(0.0)
    return Hx, Hr, D


def _order(D):
    """Greedy order: smallest sum of squared negative parts over what remains."""
    m = D.shape[0]
    P = torch.clamp(D, max=0.0) ** 2
    left = torch.ones(m, dtype=torch.float64, device=D.device)
    dead = torch.zeros(m, dtype=torch.float64, device=D.device)
    order = []
    for _ in range(m):
        c = torch.argmin(P @ left + dead)
        order.append(c)
        left[c] = 0.0
        dead[c] = math.inf
    return torch.stack(order)


def _b(E, order, M):
    m, n = E.shape
    x = E - E.mean(1, keepdim=True)
    o = order.long()
    # R of the QR of the ordered data: cov = R^T R / n, regressions from its rows
    R = torch.linalg.qr(x[o].T / math.sqrt(n), mode="r")[1]
    L = R.T * torch.sign(torch.diagonal(R))[None, :]
    Li = torch.linalg.solve_triangular(L, torch.eye(m, dtype=E.dtype, device=E.device),
                                       upper=False)
    Bp = torch.tril(-torch.diagonal(L)[:, None] * Li, -1)
    B0 = torch.zeros_like(Bp)
    B0[o[:, None], o[None, :]] = Bp
    eye = torch.eye(m, dtype=E.dtype, device=E.device)
    return B0, None if M is None else torch.stack([(eye - B0) @ Mt for Mt in M])


def exact(case, seed):
    op = case["op"]
    if op in ("bootstrap", "standard"):
        return None  # orders and counts of them
    s = _inputs(case, seed)
    if op == "var_fit":
        M, E = _var(s["X"], case["p"])
        return {"M": M, "E": E}
    if op == "measure":
        Hx, Hr, D = _measure(s["E"])
        return {"Hx": Hx, "Hr": Hr, "D": D}
    if op == "order":
        return {"order": _order(s["D"]), "gap": None}
    if op == "fit_b":
        B0, Btau = _b(s["E"], s["order"], s["M"])
        return {"B0": B0} if Btau is None else {"B0": B0, "Btau": Btau}
    if op == "batched":
        M = [_var(X, p)[0].reshape(-1) for X, (_, _, p, _) in zip(s["X"], _shapes(case, seed))]
        return {"M": torch.cat(M), "order": None, "B0": None, "Btau": None, "status": None}
    M, E = _var(s["X"], case["p"])
    D = _measure(E)[2]
    out = {"M": M, "D": D, "order": None, "B0": None, "Btau": None}
    if case["prec"] != "mixed":  # a near tie may go either way on an FP32 measure
        out["B0"], out["Btau"] = _b(E, _order(D), M)
    return out
