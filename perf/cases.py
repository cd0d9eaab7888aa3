"""The work that a user of the solver has it do, as measured cases.

Four kinds of calls, all through the public entry points of the package:

* ``solve``   -- ``Solver.solve()`` on a kept handle, then ``Solver.coeffs()``: the whole of Algorithm 2
  (points, Monte Carlo corrections along Euler paths, least-squares refit, price and deltas);
* ``iterate`` -- ``Solver.iterate(k, alpha)``: one iteration from given coefficients, with its points,
  corrections and refit handed back (checkpointing, convergence studies);
* ``readout`` -- ``Solver.eval(t, S)``: prices and deltas of the fitted surface at many scenarios;
* ``serve``   -- a batch of uneven requests through the continuous-batching ``Server``.

The seed moves the market data (spots, strike, volatility level, correlation matrix), the Monte Carlo key and
the coefficients or scenarios that a case starts from; sizes and options are the case's own.

With ``precision="mixed"`` the paths and the polynomial along them are FP32, so what a caller keeps of such a
result is FP32: corrections, coefficients, prices and deltas of mixed cases are returned as float32, the
points (always FP64) and everything of an FP64 case as float64.
"""
import itertools
import math

import numpy as np
import torch

import paper_1102_4666_gb300 as G

MASK = 0xFFFFFFFF


def _case(name, kind, **kw):
    c = {"kind": kind, "precision": "mixed", "d": 5, "vol": "sin_tanh", "a": 0.2, "rho": 0.3, "full_corr": False,
         "T": 1.0, "r": 0.03, "payoff": "put", "lam": 1.0, "half_width": 1.5, "n": 2000, "M": 1000, "N": 50,
         "eta": 3, "q": 1.0, "K_it": 10, "ls_mode": 0, "queries": 0, "requests": 0}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a one-asset European put in full FP64, the accuracy check that every user runs first
        _case("euro_d1_fp64", "solve", precision="fp64", d=1, vol="const", rho=0.0, r=0.02, lam=0.0, n=200, M=500,
              N=20, eta=4, K_it=3),
        # a one-asset American put under local volatility: a high degree, many short iterations, small kernels
        _case("american_d1", "solve", d=1, vol="abs_tanh", a=0.15, rho=0.0, r=0.02, n=1000, M=2000, N=50, eta=6,
              K_it=8),
        # the two workloads of the paper's timing tables (Section 6.4)
        _case("paper_d3", "solve", d=3, vol="const", rho=0.0, r=0.02, half_width=0.25, n=2000, M=1000, N=10),
        _case("paper_d6", "solve", d=6, vol="const", rho=0.0, r=0.02, half_width=0.25, n=2000, M=5000, N=10),
        # the American basket of five assets, degree 4
        _case("basket_d5", "solve", n=2000, M=5000, eta=4),
        # the throughput workload: the American basket of ten assets (the largest)
        _case("basket_d10", "solve", d=10, rho=0.2, n=4000, M=4000, N=100, K_it=12),
        # a desk's correlations are a matrix, not one number: ragged sizes, European call
        _case("matrix_d4", "solve", d=4, full_corr=True, payoff="call", lam=0.0, n=1501, M=1003, N=25, K_it=5),
        # a served request with a large basis (p = 924): the refit weighs as much as the paths
        _case("degree6_d5", "solve", lam=0.0, n=2801, M=1111, eta=6),
        # one FP64 iteration of ten assets from given coefficients, at the large penalty of an American option
        _case("iterate_d10_fp64", "iterate", precision="fp64", d=10, rho=0.2, lam=100.0, n=1000, M=100, N=60),
        # one iteration with the pivoted-QR refit, the paper's own choice of least squares
        _case("iterate_d5_qr", "iterate", lam=100.0, n=2000, M=1000, eta=4, ls_mode=1),
        # a hedging desk's scenario grid: prices and deltas of a fitted ten-asset surface
        _case("readout_d10", "readout", d=10, rho=0.2, n=800, M=64, N=8, queries=20000),
        # the server under a batch of uneven requests (one to ten assets, degrees 2 to 6)
        _case("serving_mix", "serve", requests=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _p(c):
    return len(_basis(c["d"] + 1, c["eta"], c["q"]))


def _cost(c):
    """Rough seconds of a pass, to keep drawn cases below the largest listed one."""
    if c["kind"] == "readout":
        return c["queries"] * _p(c) * 1e-9
    if c["kind"] == "serve":
        return 0.03 * c["requests"]
    its = c["K_it"] if c["kind"] == "solve" else 1
    p = _p(c)
    slow = c["full_corr"] or c["eta"] > (6 if c["d"] <= 5 else 4)
    path = c["N"] * c["d"] * 1e-12 + p * (1e-11 if slow else 4e-13)
    refit = 4.0 * p ** 3 * 1e-12 + (p * 3e-5 if c["ls_mode"] else 0.0)
    if c["precision"] == "fp64":
        path = c["N"] * c["d"] * 1.5e-10 + p * (1e-10 if slow else 5e-11)
        refit += c["n"] * p * p * 2e-12
    return its * (c["n"] * c["M"] * path + refit)


def draw(rng):
    while True:
        kind = rng.choice(["solve"] * 8 + ["iterate"] * 4 + ["readout"] * 2 + ["serve"])
        precision = rng.choice(["mixed", "mixed", "fp64"])
        d = rng.choice([1, 2, 3, 4, 5, 6, 7, 8, 9, 10])
        full = d >= 2 and rng.random() < 0.2
        eta = rng.randint(2, 6 if d <= 5 else 4)
        q = rng.choice([1.0, 1.0, 1.0, 0.7])
        c = _case(None, kind, precision=precision, d=d, full_corr=full, eta=eta, q=q,
                  vol=rng.choice(["const", "abs_tanh", "sin_tanh", "sin_tanh", "dupire"]),
                  a=round(rng.uniform(0.12, 0.25), 3), rho=round(rng.uniform(0.0, 0.5), 2) if d > 1 else 0.0,
                  T=round(rng.uniform(0.25, 2.0), 2), r=round(rng.uniform(0.01, 0.06), 3),
                  payoff=rng.choice(["put", "put", "call"]), n=_log_int(rng, 200, 4000), M=_log_int(rng, 100, 8000),
                  N=_log_int(rng, 10, 100), K_it=rng.randint(3, 12))
        c["lam"] = rng.choice([0.0, 1.0, 100.0] if kind == "iterate" else [0.0, 1.0])
        if kind == "iterate" and rng.random() < 0.4:
            c["ls_mode"] = 1
        if kind == "readout":
            c.update(queries=_log_int(rng, 1, 100000), M=64, N=8, n=4000, full_corr=False, lam=1.0)
        if kind == "serve":
            c.update(precision="mixed", requests=rng.randint(2, 6))
        if 3 * _p(c) <= c["n"] and 2e-4 < _cost(c) < 0.15:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _market(c, rng):
    """A workload dictionary of the package from a case and a numpy generator."""
    d, T = c["d"], c["T"]
    S0 = [float(v) for v in 100.0 * np.exp(rng.uniform(-0.03, 0.03, d))]
    K = float((95.0 if c["r"] == 0.02 and d > 1 else 100.0) * math.exp(rng.uniform(-0.02, 0.02)))
    a = float(c["a"] * rng.uniform(0.97, 1.03))
    vol = {"const": {"kind": "const", "a": a},
           "abs_tanh": {"kind": "abs_tanh", "a": a, "b": 0.1, "kappa": math.log(K)},
           "sin_tanh": {"kind": "sin_tanh", "a": a, "b": 0.05, "kappa": math.log(K)},
           "dupire": {"kind": "dupire", "s": 100.0}}[c["vol"]]
    cfg = {"d": d, "T": T, "r": c["r"], "K": K, "S0": S0, "weights": [1.0 / d] * d, "payoff": c["payoff"],
           "obstacle": "payoff", "vol": vol, "rho": c["rho"], "div": [0.0] * d, "lambda": c["lam"],
           "lo": [0.0] + [math.log(s) - c["half_width"] for s in S0],
           "hi": [T] + [math.log(s) + c["half_width"] for s in S0],
           "n": c["n"], "M": c["M"], "N": c["N"], "eta": c["eta"], "q": c["q"], "K_it": c["K_it"],
           "seed": int(rng.integers(1, 1 << 62))}
    if c["full_corr"]:  # one common factor with loadings of its own per asset, and pairwise noise
        b = rng.uniform(0.3, 0.8, d)
        F = np.concatenate([b[:, None], rng.uniform(-0.3, 0.3, (d, 2))], axis=1)
        C = F @ F.T
        s = 1.0 / np.sqrt(np.maximum(1.0, np.diag(C) + 0.1))
        C = C * s[:, None] * s[None, :]
        np.fill_diagonal(C, 1.0)
        cfg["corr"] = [[float(v) for v in row] for row in C]
    return cfg


def _start_coeffs(cfg, nu, rng):
    """Coefficients of the size that a fitted price surface has, falling with the degree."""
    deg = nu.sum(axis=1)
    return rng.standard_normal(len(nu)) * 4.0 * 0.35 ** deg + np.where(deg == 0, 8.0, 0.0)


def _request_cfgs(c, rng):
    """Requests of the serving mix: uneven dimensions, sizes and degrees."""
    out = []
    for _ in range(c["requests"]):
        d = int(rng.choice([1, 2, 5, 10]))
        n, M = int(rng.integers(300, 2000)), int(rng.integers(500, 4000))
        etas = [e for e in range(2, 7) if 3 * math.comb(d + 1 + e, e) <= n]
        rc = dict(c, d=d, n=n, M=M, N=50, K_it=10, eta=int(rng.choice(etas)), q=1.0, full_corr=False,
                  T=float(rng.uniform(0.25, 2.0)), lam=float(rng.choice([0.0, 1.0])),
                  vol="abs_tanh" if d == 1 else "sin_tanh", rho=0.3 if d > 1 else 0.0)
        out.append(_market(rc, rng))
    return out


class State:
    def __init__(self, case):
        self.kind, self.case = case["kind"], case
        self.dtype = np.float32 if case["precision"] == "mixed" else np.float64

    def out(self, **kw):
        """The results under their names, in the precision that the case computes in."""
        return {k: np.asarray(v, dtype=np.float64 if k in ("t", "x") or self.kind == "readout" else self.dtype)
                for k, v in kw.items()}


def _inputs(case, seed):
    """Everything that the seed decides: the workload dictionary and the case's own arrays."""
    rng = np.random.default_rng([seed, case["d"], case["n"]])
    if case["kind"] == "serve":
        return {"requests": _request_cfgs(case, rng)}
    cfg = _market(case, rng)
    got = {"cfg": cfg}
    if case["kind"] in ("iterate", "readout"):
        got["alpha"] = _start_coeffs(cfg, _basis(case["d"] + 1, case["eta"], case["q"]), rng)
    if case["kind"] == "readout":
        m = case["queries"]
        got["t"] = rng.uniform(0.0, case["T"], m)
        got["S"] = np.array(cfg["S0"])[None, :] * np.exp(rng.uniform(-0.4, 0.4, (m, case["d"])))
    return got


def prepare(case, seed):
    s = State(case)
    s.__dict__.update(_inputs(case, seed))
    if s.kind == "serve":
        s.server = G.Server(max_slots=16, precision=case["precision"], policy="size_lanes")
        return s
    s.solver = G.Solver(s.cfg, precision=case["precision"])
    if s.kind == "readout":
        s.solver.set_coeffs(s.alpha)
    return s


def run(s):
    if s.kind == "solve":
        rep = s.solver.solve(ls_mode=s.case["ls_mode"])
        d, k = s.case["d"], s.case["K_it"]
        # the price is the last of price_iter
        return s.out(dudx=rep.dudx[:d], price_iter=rep.price_iter[:k], resid_l2=rep.resid_l2[:k],
                     alpha=s.solver.coeffs())
    if s.kind == "iterate":
        t, x, c, alpha = s.solver.iterate(1, s.alpha, ls_mode=s.case["ls_mode"])
        return s.out(t=t, x=x, c=c, alpha=alpha)
    if s.kind == "readout":
        price, delta = s.solver.eval(s.t, s.S)
        return s.out(price=price, delta=delta)
    ids = [s.server.submit(r) for r in s.requests]
    s.server.drain()
    reps = [s.server.poll(i) for i in ids]
    return s.out(dudx=[list(r.dudx) for r in reps], price_iter=[list(r.price_iter) for r in reps])


def work(case):
    """Flops of the method: Box-Muller, correlation, volatility and Euler update of each asset and step (22, a
    transcendental counting one), the polynomial with its drift and diffusion derivatives once per path and its
    value at maturity (10 per coefficient), the symmetric normal equations.  Bytes: points, corrections, basis
    coefficients."""
    if case["kind"] == "serve":
        p = 200
        per = dict(case, d=5, n=1000, M=2000, N=50, K_it=10)
        return {"bytes": case["requests"] * 8.0 * 10 * 1000 * 7,
                "flops": case["requests"] * 10.0 * (1000.0 * 2000 * (50 * per["d"] * 22 + 10 * p) + 1000.0 * p * p)}
    d, p = case["d"], _p(case)
    if case["kind"] == "readout":
        m = case["queries"]
        return {"bytes": 8.0 * m * (2 + 2 * d) + 8.0 * p, "flops": 2.0 * m * p * (1 + d)}
    its = case["K_it"] if case["kind"] == "solve" else 1
    paths = float(case["n"]) * case["M"]
    return {"bytes": its * 8.0 * (case["n"] * (d + 2) + 2 * p),
            "flops": its * (paths * (case["N"] * d * 22.0 + 10.0 * p) + float(case["n"]) * p * p + p ** 3 / 3.0)}


# ---------------------------------------------------------------------------
# the same results in 64 bits, by torch and numpy alone
# ---------------------------------------------------------------------------

def _basis(dp, eta, q):
    """Multi-indices of total degree <= eta (q < 1: of the hyperbolic set), by degree, then lexicographically
    descending with the time variate first."""
    rows = []
    for deg in range(eta + 1):
        level = []
        for spots in itertools.combinations_with_replacement(range(dp), deg):
            nu = [0] * dp
            for v in spots:
                nu[v] += 1
            level.append(tuple(nu))
        rows += sorted(set(level), reverse=True)
    if q < 1.0:
        rows = [nu for nu in rows if sum(e ** q for e in nu if e) ** (1.0 / q) <= eta * (1 + 1e-9)]
    return np.array(rows, dtype=np.int64).reshape(-1, dp)


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK)
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c0, c1, c2, c3


def _normals(b, m, i, tag, seed):
    o = _philox(torch.full_like(m, b), m, i, torch.full_like(m, tag), seed)
    z = []
    for w0, w1 in ((o[0], o[1]), (o[2], o[3])):
        r = torch.sqrt(-2.0 * torch.log((w0.double() + 0.5) * 2.0 ** -32))
        th = (w1.double() + 0.5) * (2.0 ** -31 * math.pi)
        z += [r * torch.cos(th), r * torch.sin(th)]
    return z


def _sigma(cfg, t, x, j):
    v = cfg["vol"]
    if v["kind"] == "const":
        return torch.full_like(x, v["a"])
    if v["kind"] == "abs_tanh":
        return v["a"] + v["b"] * torch.exp(-t) * torch.tanh(x - v["kappa"]).abs()
    if v["kind"] == "sin_tanh":
        return v["a"] + v["b"] * torch.sin(j + 1 + t) * torch.tanh(x - v["kappa"])
    dev = torch.exp(x) * torch.exp(cfg["r"] * t) - v["s"]
    return 0.6 * (1.2 - torch.exp(-0.1 * t) * torch.exp(-0.001 * dev * dev)) * torch.exp(-0.05 * torch.sqrt(t))


def _payoff(cfg, X):
    s = sum(w * torch.exp(x) for w, x in zip(cfg["weights"], X))
    return torch.clamp(cfg["K"] - s if cfg["payoff"] == "put" else s - cfg["K"], min=0.0)


class _Poly:
    """u = sum_l alpha_l prod_v T_nu_lv(xi_v) on the box, its derivatives along the paths and at points."""

    def __init__(self, cfg, nu, dev):
        self.cfg, self.dev, self.dp, self.eta = cfg, dev, nu.shape[1], int(nu.max()) if nu.size else 0
        lo, hi = np.array(cfg["lo"]), np.array(cfg["hi"])
        self.ctr, self.sc = 0.5 * (lo + hi), 2.0 / (hi - lo)
        self.p = len(nu)
        act = [[(v, int(e)) for v, e in enumerate(row) if e] for row in nu]
        self.groups = []  # (function numbers, variates [F, z], table rows [F, z]) by the number z of active variates
        for z in sorted({len(a) for a in act}):
            at = [l for l, a in enumerate(act) if len(a) == z]
            var = torch.tensor([[v for v, _ in act[l]] for l in at], device=dev).reshape(len(at), z)
            row = torch.tensor([[v * (self.eta + 1) + e for v, e in act[l]] for l in at], device=dev).reshape(len(at), z)
            self.groups.append((torch.tensor(at, device=dev), var, row))
        C = torch.eye(self.dp, dtype=torch.float64, device=dev)
        C[0, 0] = 0.0
        C[1:, 1:] = torch.tensor(_corr(cfg), device=dev)
        self.C = C

    def tables(self, Y):
        """T, T', T'' of every variate and degree: [dp (eta + 1), points] each."""
        T, D, E = [], [], []
        for v in range(self.dp):
            x = (Y[v] - self.ctr[v]) * self.sc[v]
            t, d, e = [torch.ones_like(x), x], [torch.zeros_like(x), torch.ones_like(x)], [torch.zeros_like(x)] * 2
            for k in range(1, self.eta):
                t.append(2 * x * t[k] - t[k - 1])
                d.append(2 * t[k] + 2 * x * d[k] - d[k - 1])
                e.append(4 * d[k] + 2 * x * e[k] - e[k - 1])
            T += t[:self.eta + 1]
            D += d[:self.eta + 1]
            E += e[:self.eta + 1]
        return torch.stack(T), torch.stack(D), torch.stack(E)

    def blocks(self, npts):
        step = max(1, int(6e7 // max(1, npts)))
        for at, var, row in self.groups:
            for a in range(0, len(at), step):
                yield at[a:a + step], var[a:a + step], row[a:a + step]

    def matrix(self, Y):
        T, _, _ = self.tables(Y)
        B = torch.ones(self.p, Y[0].numel(), dtype=torch.float64, device=self.dev)
        for at, var, row in self.blocks(Y[0].numel()):
            for a in range(row.shape[1]):
                B[at] *= T[row[:, a]]
        return B

    def value(self, alpha, Y):
        T, _, _ = self.tables(Y)
        u = torch.zeros_like(Y[0])
        for at, var, row in self.blocks(Y[0].numel()):
            f = alpha[at][:, None].expand(-1, Y[0].numel())
            for a in range(row.shape[1]):
                f = f * T[row[:, a]]
            u += f.sum(0)
        return u

    def generator(self, alpha, Y, drift, sig):
        """u and d_t u + sum_j drift_j d_j u + 1/2 sum_jl sig_j sig_l C_jl d2_jl u."""
        T, D, E = self.tables(Y)
        n, ne = Y[0].numel(), self.eta + 1
        bt = torch.stack([torch.full_like(Y[0], self.sc[0])] + [b * self.sc[j + 1] for j, b in enumerate(drift)])
        st = torch.stack([torch.zeros_like(Y[0])] + [s * self.sc[j + 1] for j, s in enumerate(sig)])
        rep = torch.arange(self.dp, device=self.dev).repeat_interleave(ne)
        A1 = D * bt[rep] + 0.5 * E * st[rep] ** 2
        S1 = D * st[rep]
        u, g = torch.zeros_like(Y[0]), torch.zeros_like(Y[0])
        for at, var, row in self.blocks(n):
            al, z = alpha[at], row.shape[1]
            if z == 0:
                u += al.sum()
                continue
            tv = [T[row[:, a]] for a in range(z)]
            pre = tv[0]
            for a in range(1, z):
                pre = pre * tv[a]
            u += al @ pre
            for a in range(z):
                f = A1[row[:, a]]
                for c in range(z):
                    if c != a:
                        f = f * tv[c]
                g += al @ f
                sa = S1[row[:, a]]
                for b in range(a + 1, z):
                    f = sa * S1[row[:, b]]
                    for c in range(z):
                        if c not in (a, b):
                            f = f * tv[c]
                    g += (al * self.C[var[:, a], var[:, b]]) @ f
        return u, g

    def gradient(self, alpha, Y):
        """u and du/dy_v of every space variate, at a few points."""
        T, D, _ = self.tables(Y)
        u, g = torch.zeros_like(Y[0]), torch.zeros(self.dp, Y[0].numel(), dtype=torch.float64, device=self.dev)
        sc = torch.tensor(self.sc, device=self.dev)
        for at, var, row in self.blocks(Y[0].numel()):
            al, z = alpha[at], row.shape[1]
            if z == 0:
                u += al.sum()
                continue
            for a in range(z):
                f = D[row[:, a]]
                for c in range(z):
                    if c != a:
                        f = f * T[row[:, c]]
                g.index_add_(0, var[:, a], al[:, None] * f * sc[var[:, a]][:, None])
            f = T[row[:, 0]]
            for a in range(1, z):
                f = f * T[row[:, a]]
            u += al @ f
        return u, g[1:]


def _corr(cfg):
    d = cfg["d"]
    if cfg.get("corr") is not None:
        return np.array(cfg["corr"])
    return np.where(np.eye(d) > 0, 1.0, cfg["rho"])


def _points(cfg, k, dev):
    i = torch.arange(cfg["n"], device=dev)
    z, w = torch.zeros_like(i), []
    for b in range((cfg["d"] + 4) // 4):
        w += _philox(torch.full_like(i, b), i, z, torch.full_like(i, (1 << 24) | k), cfg["seed"])
    return [cfg["lo"][v] + (cfg["hi"][v] - cfg["lo"][v]) * ((w[v].double() + 0.5) * 2.0 ** -32)
            for v in range(cfg["d"] + 1)]


def _corrections(cfg, poly, alpha, k, Y, dev):
    d, N, M, T = cfg["d"], cfg["N"], cfg["M"], cfg["T"]
    L = np.linalg.cholesky(_corr(cfg))
    per = max(1, int(2e6 // M))
    got = []
    for i0 in range(0, cfg["n"], per):
        i = torch.arange(i0, min(cfg["n"], i0 + per), device=dev)
        ni = i.numel()
        m = torch.arange(M, device=dev).repeat(ni)
        i = i.repeat_interleave(M)
        ti = Y[0][i]
        X = [Y[j + 1][i] for j in range(d)]
        h = (T - ti) / N
        sq = torch.sqrt(h)
        wN = _philox(torch.zeros_like(m), m, i, torch.full_like(m, (2 << 24) | k), cfg["seed"])[0] * N
        star, theta = wN >> 32, ((wN & MASK).double() + 0.5) * 2.0 ** -32
        Xs, dX, sig_s = [None] * d, [None] * d, [None] * d
        z, b = [], 0
        for s in range(N):
            while len(z) < d:
                z += _normals(b, m, i, (3 << 24) | k, cfg["seed"])
                b += 1
            zs, z = z[:d], z[d:]
            here = star == s
            for j in range(d):
                sig = _sigma(cfg, ti + s * h, X[j], j)
                inc = sum(float(L[j, q]) * zs[q] for q in range(j + 1)) * sq
                step = (cfg["r"] - cfg["div"][j] - 0.5 * sig * sig) * h + sig * inc
                Xs[j] = X[j].clone() if s == 0 else torch.where(here, X[j], Xs[j])
                dX[j] = step if s == 0 else torch.where(here, step, dX[j])
                sig_s[j] = sig if s == 0 else torch.where(here, sig, sig_s[j])
                X[j] = X[j] + step
        zb = []
        for b in range((d + 3) // 4):
            zb += _normals(b, m, i, (4 << 24) | k, cfg["seed"])
        bb = torch.sqrt(theta * (1 - theta) * h)
        Xt = [Xs[j] + theta * dX[j] + sig_s[j] * bb * sum(float(L[j, q]) * zb[q] for q in range(j + 1))
              for j in range(d)]
        tau = ti + (star.double() + theta) * h
        drift = [cfg["r"] - cfg["div"][j] - 0.5 * sig_s[j] ** 2 for j in range(d)]
        u, gen = poly.generator(alpha, [tau] + Xt, drift, sig_s)
        uT = poly.value(alpha, [torch.full_like(tau, T)] + X)
        f = -cfg["r"] * u + cfg["lambda"] * torch.clamp(_payoff(cfg, Xt) - u, min=0.0)
        a = (T - ti) * (f + gen) + _payoff(cfg, X) - uT
        got.append(a.reshape(ni, M).mean(1))
    return torch.cat(got)


def _iteration(cfg, poly, alpha, k, dev):
    Y = _points(cfg, k, dev)
    c = _corrections(cfg, poly, alpha, k, Y, dev)
    Q, R = torch.linalg.qr(poly.matrix(Y).T.contiguous())
    step = torch.linalg.solve_triangular(R, (Q.T @ c)[:, None], upper=True)[:, 0]
    return Y, c, step


def exact(case, seed):
    if case["kind"] == "serve":
        return None  # many whole solves: over a minute
    paths = case["n"] * case["M"] * (case["K_it"] if case["kind"] == "solve" else 1.0)
    if case["kind"] != "readout" and (paths * case["N"] * case["d"] > 7e9 or paths * _p(case) > 4e10):
        return None  # over about 20 seconds
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    got = _inputs(case, seed)
    cfg, nu = got["cfg"], _basis(case["d"] + 1, case["eta"], case["q"])
    poly = _Poly(cfg, nu, dev)
    if case["kind"] == "readout":
        alpha = torch.tensor(got["alpha"], device=dev)
        S = torch.tensor(got["S"], device=dev)
        Y = [torch.tensor(got["t"], device=dev)] + [torch.log(S[:, j]) for j in range(case["d"])]
        u, g = poly.gradient(alpha, Y)
        return {"price": u, "delta": g.T / S}
    if case["kind"] == "iterate":
        alpha = torch.tensor(got["alpha"], device=dev)
        Y, c, step = _iteration(cfg, poly, alpha, 1, dev)
        return {"t": Y[0], "x": torch.stack(Y[1:]), "c": c, "alpha": alpha + step}
    alpha = torch.zeros(len(nu), dtype=torch.float64, device=dev)
    x0 = [torch.zeros(1, dtype=torch.float64, device=dev)]
    x0 += [torch.tensor([math.log(s)], dtype=torch.float64, device=dev) for s in cfg["S0"]]
    price, resid = [], []
    for k in range(cfg["K_it"]):
        _, _, step = _iteration(cfg, poly, alpha, k, dev)
        alpha = alpha + step
        resid.append(step.norm())
        u, g = poly.gradient(alpha, x0)
        price.append(u[0])
    return {"dudx": g[:, 0], "price_iter": torch.stack(price), "resid_l2": torch.stack(resid),
            "alpha": alpha}
