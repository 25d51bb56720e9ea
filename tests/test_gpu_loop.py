"""Solves whose cycle loop runs on the device against the same solves driven from the host: the same
iterates, residual histories, cycle counts and endings, bit for bit."""
import numpy as np
import pytest
import torch

from synth import grf, smoothed_grf

pytestmark = pytest.mark.gpu

SHAPE = (80, 64, 96)


def pair(gb, **opts):
    loop, host = gb.Solver(SHAPE, **opts), gb.Solver(SHAPE, **opts)
    host.set_cycle_graphs(False)
    return loop, host


def same(a, b):
    (pa, sa), (pb, sb) = a, b
    assert (sa.status, sa.cycles, sa.rel_res0, sa.rel_res) == (sb.status, sb.cycles, sb.rel_res0, sb.rel_res)
    assert sa.history == sb.history
    assert torch.equal(pa, pb)
    return sa


FLAT = [dict(prec="fp64"), dict(prec="fp64", smoother="jacobi"), dict(prec="fp64", smoother="jacobi", nu1=2, nu2=1),
        dict(prec="mixed"), dict(prec="mixed", degree=4), dict(prec="mixed", krylov=2)]


@pytest.mark.parametrize("opts", FLAT)
def test_flat_loop_equals_host_loop(gb, opts):
    F = torch.from_numpy(grf(SHAPE, 350)).cuda()
    loop, host = pair(gb, **opts)
    cycles = set()
    for tol in (1e-3, 1e-5, 1e-6, 1e-7, 1e-9):
        st = same(loop.solve(F, tol=tol), host.solve(F, tol=tol))
        assert st.status == 0 and len(st.history) == st.cycles > 0
        cycles.add(st.cycles % 2)
    assert cycles == {0, 1}                      # endings in either buffer
    guess = loop.solve(F, tol=1e-9)[0]
    for maxv in (0, 1, 2):                       # no cycle at all, and limits of either parity
        st = same(loop.solve(F, guess.clone() * 0.5, tol=0.0, max_vcycles=maxv),
                  host.solve(F, guess.clone() * 0.5, tol=0.0, max_vcycles=maxv))
        assert st.status == 4 and st.cycles == maxv
    st = same(loop.solve(F, guess.clone(), tol=1e-6), host.solve(F, guess.clone(), tol=1e-6))
    assert st.status == 0 and st.cycles == 0     # converged already


@pytest.mark.parametrize("sym", [False, True])
def test_curvilinear_loops_equal_host_loops(gb, sym):
    psi = torch.from_numpy(smoothed_grf(SHAPE, 351, 2.0, 0.4)).cuda()
    F = torch.from_numpy(grf(SHAPE, 352)).cuda()
    bar = torch.from_numpy(np.random.default_rng(353).standard_normal(SHAPE)).cuda()
    loop, host = pair(gb, op="curv", curv_sym=sym)
    cycles = set()
    for tol, maxv in ((1e-6, 100), (1e-5, 100), (1e-4, 100), (0.0, 0), (0.0, 1), (0.0, 2)):
        st = same(loop.solve(F, tol=tol, max_vcycles=maxv, psi=psi), host.solve(F, tol=tol, max_vcycles=maxv, psi=psi))
        assert st.status == (0 if tol else 4)
        cycles.add(st.cycles % 2)
        phi = torch.zeros_like(F)                # forward and transposed loops of one context in turn
        got = [s.solve_adjoint(bar, phi=phi, source=F, want_psi_bar=True, tol=tol, max_vcycles=maxv) for s in (loop, host)]
        assert got[0][2].history == got[1][2].history and got[0][2].status == got[1][2].status
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
    assert cycles == {0, 1}


@pytest.mark.parametrize("opts", [dict(prec="fp64", smoother="jacobi", omega=1.9), dict(op="curv", omega=1.9)])
def test_a_diverging_solve_ends_alike(gb, opts):
    loop, host = pair(gb, **opts)
    F = torch.from_numpy(grf(SHAPE, 354, 2.0)).cuda()
    kw = {"psi": torch.from_numpy(smoothed_grf(SHAPE, 355, 2.0, 0.4)).cuda()} if "op" in opts else {}
    st = same(loop.solve(F, tol=1e-8, max_vcycles=40, **kw), host.solve(F, tol=1e-8, max_vcycles=40, **kw))
    assert st.status == 6
    # and the next solve of the contexts starts afresh
    st = same(loop.solve(F, tol=1e-8, max_vcycles=1, **kw), host.solve(F, tol=1e-8, max_vcycles=1, **kw))
    assert st.status == 4 and st.cycles == 1


@pytest.mark.parametrize("opts", [dict(prec="fp64"), dict(prec="mixed"), dict(op="curv")])
def test_a_source_that_is_not_finite_ends_alike(gb, opts):
    loop, host = pair(gb, **opts)
    F = torch.from_numpy(grf(SHAPE, 356)).cuda()
    kw = {"psi": torch.zeros_like(F)} if "op" in opts else {}
    F[3, 4, 5] = float("inf")
    for s in (loop, host):
        _, st = s.solve(F, tol=1e-6, **kw)
        assert st.status == 5 and st.cycles == 0
