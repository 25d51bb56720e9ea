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
