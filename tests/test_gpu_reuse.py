"""One context through calls that change the basis, the read-out point, the
model, the grid and the seed in turn: every result has the bits that a context
made for that call alone gives (the basis tables and the read-out point stay on
the device and are sent again only when they change)."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu

BASE = dict(d=3, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.2, lam=0.5, n=240, M=33, N=5,
            eta=3, K_it=2, seed=5)
FULL = (np.full((3, 3), 0.3) + np.diag([0.7, 0.6, 0.65])).tolist()
SEQUENCE = [dict(), dict(S0=93.0), dict(S0=93.0, seed=6), dict(eta=2), dict(eta=4, q=0.6), dict(eta=4), dict(eta=4, n=300),
            dict(d=2, eta=4), dict(d=1, eta=6), dict(d=5, eta=2), dict(corr=FULL, eta=4), dict(eta=5, n=300), dict()]


def _run(s, graph):
    rep = s.solve(use_graph=graph)
    t = np.array([0.25, 0.5])
    price, delta = s.eval(t, np.full((2, s.cfg["d"]), 97.0))
    it = s.iterate(3, s.coeffs())
    return [np.array([rep.price] + list(rep.delta[:s.cfg["d"]])), price, delta] + [np.asarray(v) for v in it]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("graph", [0, 1])
def test_reused_context_equals_a_fresh_one(precision, graph):
    import paper_1102_4666_gb300 as G
    reused = None
    for over in SEQUENCE:
        cfg = workloads.make(**{k: v for k, v in dict(BASE, **over).items() if k != "corr"})
        cfg["corr"] = over.get("corr")
        if reused is None:
            reused = G.Solver(cfg, precision=precision)
        reused.cfg = cfg
        reused._check(reused.set_model(cfg))
        reused._check(reused.set_grid(cfg))
        fresh = G.Solver(cfg, precision=precision)
        for a, b in zip(_run(reused, graph), _run(fresh, graph)):
            assert np.array_equal(a, b), over
        fresh.close()
    want = _run(reused, graph)
    for _ in range(2):  # refused both times (16 is no degree), and the tables stay what they were
        reused.cfg = dict(cfg, eta=16)
        with pytest.raises(G.BsdeError):
            reused.solve(use_graph=graph)
        reused.cfg = cfg
        for a, b in zip(_run(reused, graph), want):
            assert np.array_equal(a, b)
    reused.close()
