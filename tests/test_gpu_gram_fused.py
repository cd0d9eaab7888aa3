"""The fused Gram kernel (bases of one 128 x 128 tile, p <= 128): the matrix
against the oracle's B^T B under the bound of test_gpu_gram.py, at the edges of
the tile, of the 8-column read-out and of the K-blocks, for several splits; and
whole solves (every matrix of a batch) against solves by QR of the same
corrections' design matrices."""
import math

import numpy as np
import pytest

import workloads
from oracle import bsde_oracle as O

pytestmark = pytest.mark.gpu


def _cfg(d, eta, n, q=1.0, K_it=1):
    return workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2},
                          rho=0.2 if d > 1 else 0.0, lam=1.0, n=n, M=96, N=3, eta=eta, K_it=K_it, seed=23, q=q)


@pytest.mark.parametrize("splits", [0, 1, 3, 4096])
@pytest.mark.parametrize("d,eta,n,q", [(1, 1, 33, 1.0), (1, 6, 200, 1.0), (2, 6, 300, 1.0), (3, 3, 2000, 1.0),
                                       (1, 14, 257, 1.0), (6, 3, 1001, 1.0), (4, 4, 600, 1.0), (10, 2, 320, 1.0)])
def test_fused_gram_against_oracle(d, eta, n, q, splits):
    import paper_1102_4666_gb300 as G
    cfg = _cfg(d, eta, n, q)
    nu = O.multi_index_set(d + 1, eta, q)
    assert len(nu) <= 128
    s = G.Solver(cfg, precision="mixed")
    A = s.gram(2, gram_splits=splits)
    s.close()
    t, x = O.points(cfg, 2)
    B = O.basis_matrix(cfg, nu, t, x)
    kblocks = (n + 31) // 32
    used = min(kblocks, splits) if splits else 1
    m = 32 * math.ceil(kblocks / used)  # the longest slice (or longer, splits 0)
    bound = (2.0 ** -20 + 3 * m * 2.0 ** -23) * (np.abs(B).T @ np.abs(B))
    assert np.all(np.abs(A - B.T @ B) <= bound)
    assert np.array_equal(A, A.T)


@pytest.mark.parametrize("d,eta,n,K_it", [(1, 6, 300, 24), (3, 3, 500, 12), (4, 3, 600, 7), (6, 3, 900, 3), (2, 2, 64, 64)])
def test_batched_matrices_refit_like_qr(d, eta, n, K_it):
    import paper_1102_4666_gb300 as G
    cfg = _cfg(d, eta, n, K_it=K_it)
    s = G.Solver(cfg, precision="mixed")
    r0 = s.solve()
    a0 = s.coeffs()
    r1 = s.solve(ls_mode=1)
    a1 = s.coeffs()
    r2 = s.solve(use_graph=0)
    a2 = s.coeffs()
    s.close()
    assert r0.status == r1.status == G.OK
    assert np.max(np.abs(a0 - a1)) <= 1e-6 * np.max(np.abs(a1))
    assert np.array_equal(a0, a2) and r0.price == r2.price
