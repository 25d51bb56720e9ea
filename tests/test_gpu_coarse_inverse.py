"""The coarsest inverse built on the GPU: the minimum-norm inverse of the coarsest operator for
4 unknowns a side and up, panel remainders and the largest size, through mg_coarse_solve."""
import numpy as np
import pytest

from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape", [(4, 4, 4), (4, 5, 6), (5, 5, 5), (7, 9, 4), (4, 8, 8), (7, 7, 7), (8, 8, 8)])
def test_coarse_solve_inverts_the_operator(gb, shape, sym):
    s = gb.Solver(shape, op="curv", levels=1, curv_sym=sym)
    assert s.levels == 1
    psi = smoothed_grf(shape, 95, 1.0, 0.4)
    s.set_geometry(torch.from_numpy(psi).cuda())
    J, _ = s.curv_geometry(0)
    J = J.double().cpu().numpy()
    rng = np.random.default_rng(96)
    u = rng.standard_normal(shape)
    u -= u.mean()
    r = s.curv_apply(0, torch.from_numpy(u).cuda(), divide_by_J=True).cpu().numpy()   # L u, in the range of L
    e = s.coarse_solve(torch.from_numpy(r).cuda()).cpu().numpy()
    # FP64 elimination: the condition number of the periodic operator on <= 8 cells a side is
    # below 1e2, times n roundings
    assert np.abs(e - u).max() <= 1e2 * u.size * 2.0 ** -52 * np.abs(u).max()
    # a right-hand side along the left null vector J gives nothing
    e = s.coarse_solve(torch.from_numpy(J).cuda()).cpu().numpy()
    assert np.abs(e).max() <= 1e2 * u.size * 2.0 ** -52 * np.abs(J).max()
    s.close()


def test_folded_mesh_is_refused(gb):
    shape = (16, 16, 16)
    s = gb.Solver(shape, op="curv")
    z = np.arange(16.0)
    psi = np.broadcast_to(40.0 * np.cos(2 * np.pi * z / 16)[:, None, None], shape).copy()
    with pytest.raises(gb.GbmgError) as e:
        s.set_geometry(torch.from_numpy(psi).cuda())
    assert e.value.status == 1
    s.set_geometry(torch.from_numpy(smoothed_grf(shape, 97, 1.5, 0.3)).cuda())   # usable afterwards
    s.close()
