"""The one-launch residual and restriction of small curvilinear levels, with the coarse level's
first sweep, inside V-cycles against the oracle (GPU)."""
import numpy as np
import pytest
import torch

from oracle import curv
from synth import grf, smoothed_grf

pytestmark = pytest.mark.gpu


# tiles of 4 x 4 x 2 coarse cells: whole; cut in x, y and z; two such levels; only the second one
@pytest.mark.parametrize("shape", [(16, 32, 24), (20, 36, 40), (36, 20, 44), (44, 36, 20), (48, 48, 48)])
@pytest.mark.parametrize("sym", [False, True])
def test_curv_vcycle_matches_oracle(gb, shape, sym):
    psi = smoothed_grf(shape, 51, 1.5, 0.4)
    s = gb.Solver(shape, op="curv", curv_sym=sym)
    s.set_geometry(torch.from_numpy(psi).cuda())
    hier = curv.hierarchy(psi, sym=sym)
    r = torch.from_numpy(grf(shape, 52)).cuda().float()
    for tr in (False, True):
        got = s.curv_vcycle(r, transpose=tr).double().cpu().numpy()
        ref = curv.vcycle(0, np.zeros(shape), r.double().cpu().numpy(), hier, transpose=tr, cache={})
        # FP32 coefficients and sweeps: about a hundred operations of 6e-8 per level, in quadrature
        assert np.linalg.norm(got - ref) <= 2e-5 * np.linalg.norm(ref)
    s.close()
