"""The z-marching curvilinear sweep and residual (levels above 64^3 cells, which a hierarchy with at
most 512 coarsest cells gives sides of a multiple of 16) and the one-cell tiles (the same for
fields off 16 bytes) against the FP64 oracle, with partial tiles in x and z runs of several
lengths; and the V-cycle above them."""
import numpy as np
import pytest

from oracle import curv
from synth import grf, smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ORDER = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape", [(80, 64, 80), (64, 96, 112), (112, 80, 64)])
def test_sweep_and_residual(gb, shape, sym):
    s = gb.Solver(shape, op="curv", curv_sym=sym)
    s.set_geometry(torch.from_numpy(smoothed_grf(shape, 361, 2.0, 0.5)).cuda())
    J, B6 = (t.double().cpu().numpy() for t in s.curv_geometry(0))
    B = np.empty((3, 3) + shape)
    for k, (a, b) in enumerate(ORDER):
        B[a, b] = B[b, a] = B6[k]
    rng = np.random.default_rng(362)
    u, r = (rng.standard_normal(shape).astype(np.float32) for _ in range(2))
    rd, aligned = torch.from_numpy(r).cuda(), torch.from_numpy(u).cuda()
    off = torch.empty(u.size + 1, device="cuda")[1:].view(shape)   # 4 bytes off: the one-cell tiles
    off.copy_(aligned)
    u, r = u.astype(np.float64), r.astype(np.float64)
    diag = curv.diag_M_sym(B, 1.0) if sym else curv.diag_M(B, 1.0)
    for tr in (False, True):
        Mu = (curv.apply_M_sym if sym else (curv.apply_MT if tr else curv.apply_M))(u, B, 1.0)
        res, sweep = r - Mu / J, u + 2.0 / 3.0 * (J * r - Mu) / diag
        for x in (aligned, off):
            # some 60 FP32 operations per cell, as in the comparisons of smaller levels
            got = s.curv_residual(0, rd, x, transpose=tr).double().cpu().numpy()
            assert np.abs(got - res).max() < 2e-5 * np.abs(res).max()
            got = s.curv_smooth(0, x, rd, transpose=tr).double().cpu().numpy()
            assert np.abs(got - sweep).max() < 2e-5 * np.abs(sweep).max()
    s.close()


@pytest.mark.parametrize("sym", [False, True])
def test_vcycle(gb, sym):
    shape = (80, 64, 80)
    psi = smoothed_grf(shape, 363, 2.0, 0.5)
    s = gb.Solver(shape, op="curv", curv_sym=sym)
    s.set_geometry(torch.from_numpy(psi).cuda())
    hier = curv.hierarchy(psi, sym=sym)
    rd = torch.from_numpy(grf(shape, 364)).float().cuda()
    for tr in (False, True):
        got = s.curv_vcycle(rd, transpose=tr).double().cpu().numpy()
        ref = curv.vcycle(0, np.zeros(shape), rd.double().cpu().numpy(), hier, transpose=tr, cache={})
        assert np.linalg.norm(got - ref) < 2e-5 * np.linalg.norm(ref)
    s.close()
