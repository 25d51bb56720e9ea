"""The one-launch residual and restriction of small levels, with the coarse level's first step,
inside FP64 V-cycles against the oracle (GPU)."""
import numpy as np
import pytest
import torch

from oracle import flat
from synth import grf

pytestmark = pytest.mark.gpu


# tiles of 4 x 4 x 2 coarse cells: whole; cut in x, y and z; the largest below and the first
# above the size from which the two kernels run
@pytest.mark.parametrize("shape", [(8, 16, 32), (20, 36, 40), (36, 20, 44), (44, 36, 20), (56, 56, 56), (64, 64, 64)])
@pytest.mark.parametrize("smoother, nu1", [("cheb", 2), ("jacobi", 0), ("jacobi", 1), ("jacobi", 2)])
def test_fp64_vcycle_matches_oracle(gb, shape, smoother, nu1):
    s = gb.Solver(shape, prec="fp64", smoother="chebyshev" if smoother == "cheb" else "jacobi", nu1=nu1)
    r = grf(shape, 9)
    got = s.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = flat.vcycle(0, np.zeros(shape), r, s.levels, smoother, nu1=nu1)
    # some hundred FP64 operations per cell and level, each 1.1e-16 of values of the result's size
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()


# the levels of at most 4096 cells in one cluster launch: 16^3 and 8^3 (a cell per thread; 32 per
# CTA), sides that leave CTAs partly or wholly empty, one smoothed level only
@pytest.mark.parametrize("shape", [(32, 32, 32), (20, 36, 40), (16, 24, 40), (64, 32, 32), (24, 24, 24)])
@pytest.mark.parametrize("degree", [1, 2, 8])
def test_fp64_bottom_chain_matches_oracle(gb, shape, degree):
    s = gb.Solver(shape, prec="fp64", degree=degree)
    r = grf(shape, 11)
    got = s.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = flat.vcycle(0, np.zeros(shape), r, s.levels, degree=degree)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
