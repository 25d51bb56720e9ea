"""The residual norm that stops a curvilinear solve, where a thread of the double-float step sums a
column of 2 x 256 squares: equal magnitudes in every cell, whose roundings a plain FP32 chain adds
up with one sign."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [False, True])
def test_norm_of_a_long_column(gb, sym):
    shape = (256, 384, 384)   # 288 tiles: one run over all planes
    i = sum(torch.arange(n, device="cuda").view([-1 if k == a else 1 for k in range(3)]) for a, n in enumerate(shape))
    sign = 1.0 - 2.0 * (i % 2).double()                      # a checkerboard: A sign = -12 sign
    f, r = float(np.float32(0.9)), float(np.float32(0.37))   # chains of 512: -2.4e-6 and +7.2e-6 of the sum
    s = gb.Solver(shape, op="curv", curv_sym=sym)
    _, st = s.solve(f * sign, (r - f) / 12.0 * sign, tol=0.0, max_vcycles=0, psi=torch.zeros(shape, dtype=torch.float64,
                                                                                            device="cuda"))
    # chains of eight squares, each addition half an ulp of at most its partial sum: 4 x 2^-24 of
    # either sum at worst, half of it on each root, together 2^-22
    assert abs(st.rel_res0 / (r / f) - 1.0) <= 2.0 ** -22
    s.close()
