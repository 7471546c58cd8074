"""A solve that stops above its tolerance is reported by the next synchronise
whatever follows it unread: eager solves, replays of the caller's graph and
replays of a batch; and it is reported once."""
import numpy as np
import pytest

from _parity import dev
from paper_2211_01185_gb300 import cfdem as cf
from paper_2211_01185_gb300 import synth

pytestmark = pytest.mark.gpu


def _case():
    return synth.make_random_case(33, n_el=(4, 5, 6), k=2, n=150, extent=(0.04, 0.05, 0.06))


def _buffers(c):
    import torch
    z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda:0")  # noqa: E731
    t = {k: dev(c[k]) for k in ("x", "r", "u_p", "u_nodal", "p_nodal")}
    return dict(t, n=c["x"].shape[0], eps=z(c["u_nodal"].shape[0]), f=z(c["x"].shape[0], 3))


def _solution(c, prm):
    """the projected void fraction, converged: a step from it needs no iteration"""
    b = _buffers(c)
    with cf.Context(c["origin"], c["extent"], c["n_el"], c["k"], dict(prm, cg_maxit=100)) as ctx:
        _step(ctx, b)
        assert cf.cfdem_synchronize(ctx.h) == cf.OK
    return b["eps"]


def _step(ctx, b):
    cf.cfdem_coupling_step(ctx.h, b["n"], b["x"], b["r"], b["u_p"], b["u_nodal"], b["p_nodal"],
                           b["eps"], b["f"])


def _reported(h):
    got = [cf.cfdem_synchronize(h, raise_on_error=False) for _ in range(2)]
    assert got[1] == cf.OK                     # once
    assert got[0] in (cf.OK, cf.NOT_CONVERGED)
    return got[0] == cf.NOT_CONVERGED


def _params(c, precision, precond=1):
    return dict(c["params"], precision=precision, cg_rtol=1e-12, cg_maxit=1, cg_precond=precond)


@pytest.mark.parametrize("precision,precond", [(0, 1), (1, 1), (0, 0)])
def test_eager_failure_then_replay_of_the_callers_graph(precision, precond):
    import torch
    c = _case()
    prm = _params(c, precision, precond)
    sol = _solution(c, prm)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        b = _buffers(c)
        with cf.Context(c["origin"], c["extent"], c["n_el"], c["k"], prm) as ctx:
            _step(ctx, b)                       # fails; from now on solves are graphed
            assert _reported(ctx.h)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=side, capture_error_mode="relaxed"):
                _step(ctx, b)
            assert not _reported(ctx.h)         # nothing ran
            b["eps"].zero_()
            _step(ctx, b)                       # fails unread
            b["eps"].copy_(sol)
            g.replay()                          # converges
            assert _reported(ctx.h)
            assert ctx.stats().converged == 1
            for rep in range(2):                # a failed replay, then one that converges
                b["eps"].zero_()
                g.replay()
                b["eps"].copy_(sol)
                g.replay()
                assert _reported(ctx.h)
            b["eps"].zero_()
            g.replay()                          # the last outcome is the failed one
            assert _reported(ctx.h)
            b["eps"].copy_(sol)
            g.replay()
            assert not _reported(ctx.h)
            b["eps"].zero_()
            g.replay()                          # fails unread
            b["eps"].copy_(sol)
            cf.cfdem_set_timing(ctx.h, 1)
            _step(ctx, b)                       # converges, with host checks
            assert _reported(ctx.h)
            assert ctx.stats().converged == 1


@pytest.mark.parametrize("precision", [0, 1])
def test_eager_failure_then_replay_of_the_batch(precision):
    import torch
    c = _case()
    prm = _params(c, precision)
    sol = _solution(c, prm)
    bh = cf.cfdem_batch_create(1, 0, torch.cuda.current_stream().cuda_stream)
    h = cf.cfdem_batch_bed(bh, 0)
    cf.cfdem_set_mesh(h, c["origin"], c["extent"], c["n_el"], c["k"])
    cf.cfdem_set_params(h, cf.make_params(**prm))
    a, b = _buffers(c), _buffers(c)

    def step(t, start):
        t["eps"].copy_(start)
        io = cf.bed_io(t["n"], t["x"], t["r"], t["u_p"], t["u_nodal"], t["p_nodal"], t["eps"],
                       t["f"])
        assert cf.cfdem_batch_coupling_step(bh, [io]) == cf.OK
        return cf.cfdem_batch_last_replayed(bh)

    zero = torch.zeros_like(sol)
    assert step(a, sol) == 0                    # eager, converges
    assert cf.cfdem_batch_synchronize(bh) == (cf.OK, -1)
    assert step(b, zero) == 0                   # other buffers: eager again, fails
    assert step(b, sol) == 1                    # replayed, converges
    assert cf.cfdem_batch_synchronize(bh) == (cf.NOT_CONVERGED, 0)
    assert cf.cfdem_batch_synchronize(bh) == (cf.OK, -1)
    assert step(b, zero) == 1 and step(b, sol) == 1
    assert cf.cfdem_batch_synchronize(bh) == (cf.NOT_CONVERGED, 0)
    assert cf.cfdem_batch_synchronize(bh) == (cf.OK, -1)
    cf.cfdem_batch_destroy(bh)
