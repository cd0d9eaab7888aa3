"""The coefficients of one iteration against the oracle's normal equations with
the same points and the GPU's own corrections, on both sides of the rules that
choose how A^-1 is applied (as one matrix, or as the two triangular factors for
large bases with fresh points), in both precisions and for fixed points.

Bound: the last refinement step leaves a relative error of the preconditioner's
times that of the step before, and the FP64 residual one of cond(A) 2^-53 per
step; cond(A) of these Chebyshev bases with n >= 2 p uniform points is below
1e6, hence 1e-9 of the largest coefficient change."""
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
