"""mg_curv_smooth on the coarsest level, which the V-cycle itself never smooths, against the FP64
oracle: hierarchies of several levels and of one, a given iterate and a zero one."""
import numpy as np
import pytest

from oracle import curv
from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ORDER = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape,levels", [((16, 16, 16), 0), ((40, 24, 20), 0), ((4, 4, 4), 1), ((7, 5, 6), 1)])
def test_sweep_of_the_coarsest_level(gb, shape, levels, sym):
    s = gb.Solver(shape, op="curv", levels=levels, curv_sym=sym)
    s.set_geometry(torch.from_numpy(smoothed_grf(shape, 61, 1.0, 0.4)).cuda())
    level = s.levels - 1
    h = 2.0 ** level
    J, B6 = (t.double().cpu().numpy() for t in s.curv_geometry(level))
    B = np.empty((3, 3) + J.shape)
    for k, (a, b) in enumerate(ORDER):
        B[a, b] = B[b, a] = B6[k]
    rng = np.random.default_rng(62)
    r = rng.standard_normal(J.shape).astype(np.float32)
    e = rng.standard_normal(J.shape).astype(np.float32)
    diag = curv.diag_M_sym(B, h) if sym else curv.diag_M(B, h)
    for tr in (False, True):
        op = curv.apply_M_sym if sym else (curv.apply_MT if tr else curv.apply_M)
        for u in (None, e):
            u64 = np.zeros(J.shape) if u is None else u.astype(np.float64)
            ref = u64 + 2.0 / 3.0 * (J * r - op(u64, B, h)) / diag
            got = s.curv_smooth(level, None if u is None else torch.from_numpy(u).cuda(),
                                torch.from_numpy(r).cuda(), transpose=tr).double().cpu().numpy()
            # some 60 FP32 operations per cell, each off by 2^-24 of a term no larger than a few
            # times the largest value: below 2e-5 of it, as on the finer levels
            assert np.abs(got - ref).max() < 2e-5 * np.abs(ref).max()
    s.close()
