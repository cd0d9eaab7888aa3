"""Contexts of several host threads at the same time, with bases that need
shared memory of different sizes from the same kernels: every call succeeds and
gives the bits of the same call made alone."""
import threading

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _cfg(d, eta, n, **kw):
    return workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2},
                          rho=0.3 if d > 1 else 0.0, lam=0.5, n=n, M=33, N=5, eta=eta, K_it=2, seed=9, **kw)


def _together(jobs, rounds):
    """Every job `rounds` times in a thread of its own; results other than the one it gives alone."""
    want = [job() for job in jobs]
    gate, bad = threading.Barrier(len(jobs)), []

    def loop(job, first):
        gate.wait()
        for _ in range(rounds):
            try:
                got = job()
                if not all(np.array_equal(a, b) for a, b in zip(got, first)):
                    bad.append("other bits")
            except Exception as e:  # noqa: BLE001
                bad.append(repr(e))

    threads = [threading.Thread(target=loop, args=v) for v in zip(jobs, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return bad


def test_read_outs_of_different_bases():
    import paper_1102_4666_gb300 as G
    rng = np.random.default_rng(2)
    solvers, jobs = [], []
    for d, eta, n in [(10, 3, 800), (1, 2, 40), (5, 6, 2000), (2, 12, 1000)]:
        s = G.Solver(_cfg(d, eta, n), precision="fp64")
        s.solve(use_graph=0)
        m = 1300
        t, S = rng.uniform(0.0, 1.0, m), 100.0 * np.exp(rng.uniform(-0.5, 0.5, (m, d)))
        solvers.append(s)
        jobs.append(lambda s=s, t=t, S=S: s.eval(t, S))
    bad = _together(jobs, 400)
    for s in solvers:
        s.close()
    assert bad == []


@pytest.mark.parametrize("precision,bases", [("fp64", [(5, 6, 2000), (6, 3, 400), (3, 7, 800)]),
                                             ("mixed", [(2, 14, 1500), (3, 8, 1100), (2, 9, 500)])])
def test_solves_of_different_bases(precision, bases):
    import paper_1102_4666_gb300 as G
    solvers = [G.Solver(_cfg(d, eta, n), precision=precision) for d, eta, n in bases]

    def job(s):
        rep = s.solve(use_graph=0, check=True, allow_underdetermined=1)
        return np.array([rep.price]), s.coeffs()

    bad = _together([lambda s=s: job(s) for s in solvers], 40)
    for s in solvers:
        s.close()
    assert bad == []
