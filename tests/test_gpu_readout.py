"""Price and deltas at many points (Solver.eval) against the oracle's
evaluation of the same coefficients: query counts at the edges of the kernel's
groups of 32 and of its split over basis functions, degrees and dimensions at
both ends, hyperbolic bases, prices far from the box, deltas left out."""
import ctypes

import numpy as np
import pytest

import workloads
from oracle import bsde_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,eta,q,m", [(1, 1, 1.0, 1), (1, 6, 1.0, 33), (2, 15, 1.0, 31), (3, 0, 1.0, 5), (4, 5, 0.7, 64),
                                       (5, 6, 1.0, 257), (10, 3, 1.0, 40000), (10, 4, 1.0, 3), (10, 5, 0.6, 100),
                                       (3, 2, 1.0, 1249), (5, 6, 0.8, 2000), (10, 2, 1.0, 1217), (2, 0, 1.0, 3000)])
def test_eval_against_oracle(d, eta, q, m):
    import paper_1102_4666_gb300 as G
    n = 2 * len(O.multi_index_set(d + 1, eta, q)) + 2
    cfg = workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.0, lam=0.0,
                         n=n, M=2, N=2, eta=eta, K_it=1, seed=3, q=q)
    nu = O.multi_index_set(d + 1, eta, q)
    rng = np.random.default_rng(8)
    alpha = rng.standard_normal(len(nu)) / (1.0 + nu.sum(axis=1)) ** 2
    t = rng.uniform(0.0, 1.0, m)
    S = 100.0 * np.exp(rng.uniform(-1.5, 1.5, (m, d)))
    S[0] = 100.0 * np.exp(1.6)  # just outside the box
    s = G.Solver(cfg, precision="fp64")
    s.set_coeffs(alpha)
    price, delta = s.eval(t, S)
    only = np.zeros(m)
    dp = ctypes.POINTER(ctypes.c_double)
    assert G.bsde_eval_price_delta(s.h, m, t.ctypes.data_as(dp), S.ctypes.data_as(dp), only.ctypes.data_as(dp), None) == G.OK
    bad = S.copy()
    bad[-1, -1] = 0.0
    with pytest.raises(G.BsdeError):
        s.eval(t, bad)
    s.close()
    assert np.array_equal(only, price)
    pick = np.unique(np.concatenate([np.arange(min(m, 40)), [m - 1], rng.integers(0, m, 20)]))
    u, g = O.eval_u(cfg, nu, alpha, t[pick], np.log(S[pick]).T)
    g = g.T / S[pick] if d > 0 and len(g) else np.zeros((len(pick), d))
    assert np.max(np.abs(price[pick] - u)) <= 1e-9 * max(1e-300, np.max(np.abs(u)))
    if eta > 0:
        assert np.max(np.abs(delta[pick] - g)) <= 1e-9 * np.max(np.abs(g))
