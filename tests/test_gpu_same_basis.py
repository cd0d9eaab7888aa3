"""Coefficients stay with a context while the basis keeps its functions, also
under another exponent q of the hyperbolic set: a resumed solve and an iteration
from the current coefficients go on from them, and the surface can be read."""
import numpy as np
import pytest

import workloads
from oracle import bsde_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,eta,q0,q1", [(3, 1, 1.0, 0.5), (2, 3, 0.7, 0.72), (4, 4, 0.5, 0.52), (1, 0, 1.0, 0.3)])
def test_another_q_with_the_same_functions(d, eta, q0, q1):
    import paper_1102_4666_gb300 as G
    assert np.array_equal(O.multi_index_set(d + 1, eta, q0), O.multi_index_set(d + 1, eta, q1))
    cfg = workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.2 if d > 1 else 0.0,
                         lam=0.5, n=200, M=33, N=5, eta=eta, K_it=2, seed=5, q=q0)
    s = G.Solver(cfg, precision="fp64")
    s.solve()
    a0 = s.coeffs()
    want = s.iterate(2)[3]
    s.cfg = dict(cfg, q=q1)
    s.set_coeffs(a0)
    s.cfg = dict(cfg, q=q0)
    assert np.array_equal(s.iterate(2)[3], want)
    s.set_coeffs(a0)
    s.cfg = dict(cfg, q=q1)
    assert np.array_equal(s.iterate(2)[3], want)
    s.cfg = dict(cfg, q=q0)
    s.solve(k_start=3, K_it=1)
    s.close()


def test_another_q_with_other_functions_starts_anew():
    import paper_1102_4666_gb300 as G
    cfg = workloads.make(d=2, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.2, lam=0.5,
                         n=200, M=33, N=5, eta=3, K_it=2, seed=5)
    s = G.Solver(cfg, precision="fp64")
    s.solve()
    s.cfg = dict(cfg, q=0.5)
    with pytest.raises(G.BsdeError):
        s.solve(k_start=2, K_it=1)
    s.close()
