"""Solves at the limits of device memory: the partial sums of the path kernel
take no more than four rounds of paths per CTA (256 FP64 or 512 FP32 paths)
need where a budget or the allocator has no room for more, and a grid that no
launch can have is refused."""
import re

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
FULL = [[1.0, 0.3, 0.1], [0.3, 1.0, 0.5], [0.1, 0.5, 1.0]]


def _cfg(d=2, n=320, M=4096, eta=3, **kw):
    corr = kw.pop("corr", None)
    cfg = workloads.make(d=d, T=1.0, r=0.03, K=100.0, S0=100.0, vol={"kind": "const", "a": 0.2}, rho=0.2, lam=0.5, n=n, M=M,
                         N=2, eta=eta, K_it=2, seed=5, **kw)
    cfg["corr"] = corr
    return cfg


def _needs(cfg, precision, **kw):
    """Bytes of the smallest budget, as the refusal of a smaller one states them."""
    import paper_1102_4666_gb300 as G
    s = G.Solver(cfg, precision=precision, mem_budget=1)
    with pytest.raises(G.BsdeError) as e:
        s.solve(**kw)
    s.close()
    return int(re.search(r"needs (\d+) bytes", str(e.value)).group(1))


@pytest.mark.parametrize("precision,eta,per,tol", [("fp64", 3, 256, 1e-10), ("fp64", 7, 256, 1e-10), ("mixed", 3, 512, 1e-5),
                                                   ("mixed", 7, 512, 1e-5)])
def test_partial_sums_within_a_budget(precision, eta, per, tol):
    import paper_1102_4666_gb300 as G
    cfg = _cfg(eta=eta)
    need = _needs(cfg, precision)
    assert need - _needs(_cfg(eta=eta, M=per), precision) <= cfg["n"] * 8 * (cfg["M"] // per - 1)
    s, free = G.Solver(cfg, precision=precision, mem_budget=need), G.Solver(cfg, precision=precision)
    a, b = s.solve(), free.solve()
    assert abs(a.price - b.price) <= tol * abs(b.price)
    assert s.solve().price == a.price
    s.close()
    free.close()
    # the server reckons with 256 paths per CTA in FP64, the context came down to 512
    srv = G.Server(max_slots=2, precision=precision, mem_budget=need + cfg["n"] * 8 * 8)
    i = srv.submit(cfg)
    srv.drain()
    assert abs(srv.poll(i).price - b.price) <= tol * abs(b.price)
    srv.close()


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("mixed", 1e-4)])
def test_full_correlation_in_the_memory_of_its_tables(precision, tol):
    """The monomial form takes some kilobytes more than the per-thread tables."""
    import paper_1102_4666_gb300 as G
    cfg = _cfg(d=3, M=100, corr=FULL)
    s = G.Solver(cfg, precision=precision, mem_budget=_needs(cfg, precision, eval_mode=1))
    free = G.Solver(cfg, precision=precision)
    a, b = s.solve(), free.solve()
    s.close()
    free.close()
    assert abs(a.price - b.price) <= tol * abs(b.price)


def test_many_partial_sums():
    """Above 64 MB the partial sums are those of four rounds, whatever the budget: the extra
    memory of the faster shapes stays small beside what a device has free."""
    import paper_1102_4666_gb300 as G
    for precision, per, eta in (("fp64", 256, 1), ("fp64", 256, 7), ("mixed", 512, 1)):
        n, M, held = 3200, 2**20, []
        s = G.Solver(_cfg(n=n, M=M, eta=eta), precision=precision, allocator=_Refusing(held))
        assert s.solve(check=False).status == G.ERR_NOMEM
        s.close()
        assert held[0] <= max(64 << 20, n * 8 * (M // per)) + (8 << 20), (precision, eta, held)


class _Refusing:
    """An allocator that has nothing, and notes what it was asked for."""

    def __init__(self, asked):
        self.asked = asked

    def alloc(self, nbytes, stream):
        self.asked.append(nbytes)
        return None

    def free(self, ptr, stream):
        pass


def test_more_ctas_than_a_grid_holds():
    import paper_1102_4666_gb300 as G
    cfg = _cfg(n=4000, M=2**31 - 1, eta=1)
    for precision in ("fp64", "mixed"):
        s = G.Solver(cfg, precision=precision)
        with pytest.raises(G.BsdeError) as e:
            s.solve()
        assert "2^31" in str(e.value)
        s.close()
