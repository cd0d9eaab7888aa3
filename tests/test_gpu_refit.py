"""The coefficients of one iteration against the oracle's normal equations with
the same points and the GPU's own corrections, on both sides of the rules that
choose how A^-1 is applied (as one matrix, or as the two triangular factors for
large bases with fresh points), in both precisions and for fixed points.

Bound: a refinement step multiplies the error by cond(A) times the relative error
of the Gram matrix (2^-24 in mixed precision, two steps; 2^-53 in FP64, one); the
bases and counts here have cond(A) below 1e4, so (6e-4)^3 = 2e-10 of the largest
coefficient change, and 1e-9 is asked for."""
import numpy as np
import pytest

import workloads
from oracle import bsde_oracle as O

pytestmark = pytest.mark.gpu


def _iterate(d, eta, n, precision, resample, q=1.0, **kw):
    import paper_1102_4666_gb300 as G
    cfg = workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.1, lam=0.0,
                         n=n, M=4, N=2, eta=eta, K_it=3, seed=7, q=q)
    nu = O.multi_index_set(d + 1, eta, q)
    a0 = np.zeros(len(nu))
    a0[0] = 5.0
    s = G.Solver(cfg, precision=precision)
    s._check(s.set_grid(cfg, resample=resample))
    t, x, c, a1 = s.iterate(2, a0, **kw)
    s.solve(use_graph=0)
    by_solve = s.coeffs()
    s.solve(use_graph=1)
    graph = s.coeffs()
    a = np.zeros(len(nu))
    for k in range(3):
        _, _, _, a = s.iterate(k, a)
    s.close()
    assert np.array_equal(by_solve, a) and np.array_equal(graph, a)
    B = O.basis_matrix(cfg, nu, t, x)
    delta = np.linalg.lstsq(B, c, rcond=None)[0]
    assert np.max(np.abs(a1 - a0 - delta)) <= 1e-9 * np.max(np.abs(delta))


# p = 286 and 364 (below and above the line of FP64 with one refinement, p = 330),
# 364 and 495 (of mixed with two, p = 378), p = 220 with many refinements
@pytest.mark.parametrize("d,eta,n,precision,resample,kw", [
    (9, 3, 700, "fp64", 1, {}), (10, 3, 731, "fp64", 1, {}), (10, 3, 731, "fp64", 0, {}), (10, 3, 750, "mixed", 1, {}),
    (7, 4, 1003, "mixed", 1, {}), (7, 4, 1003, "mixed", 0, {}), (8, 3, 450, "mixed", 1, dict(refine_steps=9)),
    (10, 3, 731, "fp64", 1, dict(refine_steps=4))])
def test_large_basis(d, eta, n, precision, resample, kw):
    _iterate(d, eta, n, precision, resample, **kw)


# bases refitted in one launch: the smallest and the largest of the rule (p = 56
# and 66 on both sides of 64, n (p + 1) = 150000 and beyond), sizes that leave the last
# of 15 blocks of points short or empty, many
# refinements
@pytest.mark.parametrize("d,eta,n,precision,resample,q,kw", [
    (1, 0, 2, "fp64", 1, 1.0, {}), (1, 1, 7, "mixed", 1, 1.0, {}), (1, 4, 200, "fp64", 1, 1.0, {}), (1, 6, 1000, "mixed", 1, 1.0, {}),
    (1, 9, 600, "mixed", 0, 1.0, {}), (1, 10, 700, "fp64", 1, 1.0, {}), (4, 3, 1501, "mixed", 1, 1.0, {}),
    (4, 3, 2631, "mixed", 1, 1.0, {}), (4, 3, 2632, "mixed", 1, 1.0, {}), (1, 0, 16384, "mixed", 1, 1.0, {}), (1, 1, 16385, "mixed", 1, 1.0, {}),
    (2, 7, 1311, "fp64", 1, 0.6, {}), (5, 2, 5172, "mixed", 1, 1.0, dict(refine_steps=5)),
    (3, 3, 2000, "mixed", 1, 1.0, dict(refine_steps=2)), (6, 3, 300, "mixed", 1, 1.0, {})])
def test_small_basis(d, eta, n, precision, resample, q, kw):
    _iterate(d, eta, n, precision, resample, q, **kw)


def test_small_basis_launches_and_resume():
    """Three launches an iteration beside the factors, and a solve resumed from
    its own coefficients (another split into calls, another first iteration)."""
    import paper_1102_4666_gb300 as G
    cfg = workloads.make(d=3, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.1, lam=10.0,
                         n=500, M=40, N=5, eta=3, K_it=7, seed=7)
    s = G.Solver(cfg)
    seven = s.solve().kernel_launches
    want = s.coeffs()
    assert s.solve(K_it=6).kernel_launches == seven - 3
    s.solve(K_it=4, use_graph=0)
    rep = s.solve(K_it=3, k_start=4)
    assert np.array_equal(s.coeffs(), want)
    price, _ = s.eval(np.zeros(1), np.full((1, 3), 100.0))
    assert abs(price[0] - rep.price) <= 1e-12 * rep.price
    s.close()
