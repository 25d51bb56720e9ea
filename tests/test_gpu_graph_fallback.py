"""Graphs whose construction fails (here on request, at the end of the loop's capture): the solve
goes on without them, with the same results, and so do later ones."""
import numpy as np
import pytest
import torch

from synth import grf, smoothed_grf

pytestmark = pytest.mark.gpu

SHAPE = (32, 48, 64)


@pytest.mark.parametrize("prec,krylov", [("fp64", 0), ("mixed", 0), ("mixed", 2)])
def test_flat_solve_without_its_loop(gb, prec, krylov):
    F = torch.from_numpy(grf(SHAPE, 320)).cuda()
    eager, refused = (gb.Solver(SHAPE, prec=prec, krylov=krylov) for _ in range(2))
    eager.set_cycle_graphs(False)
    gb._check(gb.lib().mg_set_cycle_graphs(refused._c(), gb.TEST_REFUSE))
    for tol in (1e-9, 1e-4):
        pe, se = eager.solve(F, tol=tol)
        pr, sr = refused.solve(F, tol=tol)
        assert sr.status == se.status == 0 and sr.history == se.history
        assert torch.equal(pr, pe)
    assert gb.lib().mg_last_error() == b""
    refused.set_cycle_graphs(True)
    pr, sr = refused.solve(F, tol=1e-4)
    assert sr.cycles == se.cycles and torch.equal(pr, pe)


@pytest.mark.parametrize("sym", [False, True])
def test_curvilinear_solve_without_its_loop(gb, sym):
    psi = torch.from_numpy(smoothed_grf(SHAPE, 321, 2.0, 0.4)).cuda()
    F = torch.from_numpy(grf(SHAPE, 322)).cuda()
    bar = torch.from_numpy(np.random.default_rng(323).standard_normal(SHAPE)).cuda()
    eager, refused = (gb.Solver(SHAPE, op="curv", curv_sym=sym) for _ in range(2))
    eager.set_cycle_graphs(False)
    gb._check(gb.lib().mg_set_cycle_graphs(refused._c(), gb.TEST_REFUSE))
    for tol in (1e-7, 1e-4):
        got = []
        for s in (eager, refused):
            phi, st = s.solve(F, tol=tol, max_vcycles=100, psi=psi)
            d, p, sa = s.solve_adjoint(bar, phi=phi, source=F, want_psi_bar=True, tol=tol, max_vcycles=100)
            got.append((phi, d, p, st.history, sa.history))
        assert got[0][3:] == got[1][3:]
        assert all(torch.equal(a, b) for a, b in zip(got[0][:3], got[1][:3]))


@pytest.mark.parametrize("refusal", ["TEST_REFUSE", "TEST_REFUSE_INSTANTIATE"])
@pytest.mark.parametrize("degree", [1, 3])
def test_batch_without_its_phase_graph(gb, degree, refusal):
    shapes = [(32, 32, 32), (64, 48, 64)]
    F = [torch.from_numpy(grf(s, 324 + i)).cuda() for i, s in enumerate(shapes)]
    batch = gb.Batch(shapes, degree=degree)
    got = []
    for mode in (0, getattr(gb, refusal), getattr(gb, refusal)):
        gb._check(gb.lib().mg_batch_use_graph(batch._b, mode))
        phi = [torch.zeros_like(f) for f in F]
        stats, _ = batch.solve(F, phi, tol=1e-8)
        got.append((phi, [s.history for s in stats]))
    for phi, hist in got[1:]:
        assert hist == got[0][1]   # (the phase graph sums the norms over other tiles)
        assert all(torch.equal(a, b) for a, b in zip(phi, got[0][0]))
    batch.close()
