"""The FP64 bottom where a cluster of 16 CTAs is refused (here on request): the launches that the
cluster kernel replaces, with the same bits."""
import pytest
import torch

from synth import grf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,degree", [((32, 32, 32), 3), ((24, 40, 16), 1), ((64, 32, 48), 8)])
def test_bottom_without_a_cluster(gb, shape, degree):
    F = torch.from_numpy(grf(shape, 340)).cuda()
    got = []
    for refuse in (False, True):
        s = gb.Solver(shape, prec="fp64", degree=degree)
        s.set_cycle_graphs(False)
        if refuse:
            gb._check(gb.lib().mg_set_cycle_graphs(s._c(), gb.TEST_REFUSE))
        n = gb.launch_count()
        e = s.vcycle(F)
        n = gb.launch_count() - n
        phi, st = s.solve(F, tol=1e-9)
        got.append((e, phi, n, st.cycles))
    (ea, pa, na, ca), (eb, pb, nb, cb) = got
    assert nb > na          # (the cluster launch is the form that runs where it fits)
    assert torch.equal(ea, eb) and torch.equal(pa, pb) and ca == cb
