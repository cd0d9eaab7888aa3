"""The dense evaluation of u^k for a full correlation matrix (total degree
<= 3 at any d, <= 4 at d <= 5) against the oracle, teacher-forced, and against
the per-thread Chebyshev tables that it takes the place of; tolerances as in
test_gpu_parity.py."""
import numpy as np
import pytest

import workloads
from oracle import bsde_oracle as O
from test_gpu_parity import MIXED_C_TOL, _alpha, _nu, _scale, rel

pytestmark = pytest.mark.gpu


def _cfg(d, eta, q=1.0, vol="sin_tanh", payoff="put"):
    rng = np.random.default_rng(100 * d + eta)
    F = rng.uniform(-0.7, 0.7, (d, 3))
    C = F @ F.T
    s = 1.0 / np.sqrt(np.diag(C) + 0.5)
    C = C * s[:, None] * s[None, :]
    np.fill_diagonal(C, 1.0)
    cfg = workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0,
                         vol={"kind": vol, "a": 0.2, "b": 0.05, "kappa": workloads.LOG100, "s": 100.0}, rho=0.0,
                         lam=1.0, n=2 * workloads.basis_size(d, eta) + 3, M=37, N=5, eta=eta, K_it=1, seed=17, q=q,
                         payoff=payoff)
    cfg["corr"] = C.tolist()
    return cfg


CASES = [(2, 3, 1.0, "sin_tanh", "put"), (3, 4, 1.0, "dupire", "call"), (4, 3, 1.0, "abs_tanh", "put"),
         (5, 4, 1.0, "sin_tanh", "put"), (5, 4, 0.8, "const", "call"), (6, 3, 1.0, "const", "put"),
         (7, 2, 1.0, "sin_tanh", "put"), (8, 3, 0.7, "abs_tanh", "put"), (9, 1, 1.0, "dupire", "put"),
         (10, 3, 1.0, "sin_tanh", "put")]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "d%d-deg%d-q%g-%s-%s" % c)
def test_full_correlation_iteration(case, precision):
    import paper_1102_4666_gb300 as G
    cfg = _cfg(*case)
    nu = _nu(cfg)
    a0 = _alpha(cfg, nu)
    want = O.iteration(cfg, nu, a0, 1)
    s = G.Solver(cfg, precision=precision)
    for mode in (0, 1):  # the dense form, the tables
        t, x, c, a1 = s.iterate(1, a0, eval_mode=mode)
        if precision == "fp64":
            assert rel(c, want["c"]) < 1e-9 and rel(a1, want["alpha"]) < 1e-9
        else:
            assert np.max(np.abs(c - want["c"])) <= MIXED_C_TOL * _scale(cfg, nu, a0, t, x)
    with pytest.raises(G.BsdeError):  # asked for by name the dense form still needs a constant correlation
        s.iterate(1, a0, eval_mode=2)
    s.close()
