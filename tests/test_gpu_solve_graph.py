"""Eager solves keep their CG loop as a graph from the second solve on: the
results and statistics stay those of the first solve, failures are reported
whichever solve they come from, and changes of parameters and mesh, captures
and other contexts in between are followed."""
import numpy as np
import pytest

from _parity import dev, host
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


def _case(k, n_el=(4, 5, 6)):
    return synth.make_random_case(31 + k, n_el=n_el, k=k, n=150, extent=(0.04, 0.05, 0.06))


class _Step:
    def __init__(self, c, stream=None, **prm):
        import torch
        self.c, self.n = c, c["x"].shape[0]
        self.ctx = cf.Context(c["origin"], c["extent"], c["n_el"], c["k"],
                              dict(c["params"], **prm), stream=stream)
        self.t = [dev(c[k]) for k in ("x", "r", "u_p", "u_nodal", "p_nodal")]
        z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda:0")  # noqa: E731
        self.eps, self.f = z(c["u_nodal"].shape[0]), z(self.n, 3)
        torch.cuda.synchronize()

    def run(self):
        self.eps.zero_()
        x, r, up, u, p = self.t
        cf.cfdem_coupling_step(self.ctx.h, self.n, x, r, up, u, p, self.eps, self.f)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 3])
def test_later_solves_give_the_first_ones_bits(k, precision):
    a = _Step(_case(k), precision=precision, cg_rtol=1e-13 if precision == 0 else 1e-12)
    first = None
    for rep in range(4):
        a.run()
        cf.cfdem_synchronize(a.ctx.h)
        s = a.ctx.stats()
        got = (host(a.eps), host(a.f), s.cg_iterations, s.cg_relres, s.converged)
        if first is None:
            first = got
            assert s.converged == 1 and s.cg_iterations >= 1
        for u, v in zip(first, got):
            assert np.array_equal(u, v)
    # a warm start converges at once
    cf.cfdem_project(a.ctx.h, None, a.eps)
    cf.cfdem_synchronize(a.ctx.h)
    assert a.ctx.stats().cg_iterations <= 1


@pytest.mark.parametrize("precision", [0, 1])
def test_failures_are_reported(precision):
    a = _Step(_case(2), precision=precision, cg_rtol=1e-12, cg_maxit=1)
    for rep in range(3):                       # one iteration is not enough
        a.run()
        assert cf.cfdem_synchronize(a.ctx.h, raise_on_error=False) == cf.NOT_CONVERGED
        assert a.ctx.stats().converged == 0 and a.ctx.stats().cg_iterations == 1
        assert cf.cfdem_synchronize(a.ctx.h, raise_on_error=False) == cf.OK
    # a failure followed by a solve that converges, nothing read in between:
    # the right-hand side of a constant void fraction is solved from itself
    a.run()
    cf.cfdem_project(a.ctx.h, None, a.eps)     # closer, still failing
    sol = a.eps.clone()
    b = _Step(_case(2), precision=precision, cg_rtol=1e-12)
    b.run()
    sol.copy_(b.eps)
    cf.cfdem_synchronize(b.ctx.h)
    cf.cfdem_project(a.ctx.h, None, sol)       # starts at the solution: converged
    assert cf.cfdem_synchronize(a.ctx.h, raise_on_error=False) == cf.NOT_CONVERGED
    assert a.ctx.stats().converged == 1
    assert cf.cfdem_synchronize(a.ctx.h, raise_on_error=False) == cf.OK
    # a failure judged by its own tolerance, not by one set afterwards
    a.run()
    a.ctx.set_params(dict(a.c["params"], precision=precision, cg_rtol=0.5))
    assert cf.cfdem_synchronize(a.ctx.h, raise_on_error=False) == cf.NOT_CONVERGED


@pytest.mark.parametrize("precision", [0, 1])
def test_configuration_changes_and_other_contexts(precision):
    import torch
    c1, c2 = _case(2), _case(1, (6, 4, 5))
    tol = 1e-13 if precision == 0 else 1e-12
    ref = {}
    for name, c, l2 in (("a", c1, None), ("b", c1, 3e-5), ("c", c2, None)):
        prm = dict(precision=precision, cg_rtol=tol)
        if l2 is not None:
            prm["l2_smoothing"] = l2
        s = _Step(c, **prm)
        s.run()
        cf.cfdem_synchronize(s.ctx.h)
        ref[name] = host(s.eps)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        a = _Step(c1, precision=precision, cg_rtol=tol)
        o = _Step(c2, precision=precision, cg_rtol=tol)
        for rep in range(3):
            a.run()
            o.run()
        side.synchronize()
        assert np.array_equal(host(a.eps), ref["a"]) and np.array_equal(host(o.eps), ref["c"])
        a.ctx.set_params(dict(c1["params"], precision=precision, cg_rtol=tol, l2_smoothing=3e-5))
        for rep in range(3):
            a.run()
        side.synchronize()
        assert np.array_equal(host(a.eps), ref["b"])
        # the same context captured by the caller, then eager again
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side, capture_error_mode="relaxed"):
            a.run()
        a.eps.fill_(7.0)
        g.replay()
        side.synchronize()
        assert np.array_equal(host(a.eps), ref["b"])
        a.run()
        side.synchronize()
        assert np.array_equal(host(a.eps), ref["b"])
        # another mesh on the same context
        cf.cfdem_set_mesh(a.ctx.h, c2["origin"], c2["extent"], c2["n_el"], c2["k"])
        a.ctx.set_params(dict(c2["params"], precision=precision, cg_rtol=tol))
        o.eps.zero_()
        for rep in range(3):
            o.eps.zero_()
            x, r, up, u, p = o.t
            cf.cfdem_coupling_step(a.ctx.h, o.n, x, r, up, u, p, o.eps, o.f)
        side.synchronize()
        assert np.array_equal(host(o.eps), ref["c"])
        cf.cfdem_synchronize(a.ctx.h)
