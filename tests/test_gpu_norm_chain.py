"""The residual norm of a mixed flat solve on a mesh whose finest level is cut into chunks of 64
planes: equal magnitudes in every cell, whose roundings an FP32 chain adds up with one sign."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_norm_of_a_long_chunk(gb):
    shape = (320, 320, 160)
    i = sum(torch.arange(n, device="cuda").view([-1 if k == a else 1 for k in range(3)]) for a, n in enumerate(shape))
    sign = 1.0 - 2.0 * (i % 2).double()                      # a checkerboard: A sign = -12 sign
    f, r = float(np.float32(1.91)), float(np.float32(1.27))  # chains of 256: -3.3e-6 and +3.5e-6 of the sum
    s = gb.Solver(shape)
    _, st = s.solve(f * sign, (r - f) / 12.0 * sign, tol=0.0, max_vcycles=0)
    # chains of 32 squares, each addition half an ulp of at most its partial sum: 16 x 2^-24 of
    # either sum, half of it on each root; the residual rounded to FP32 once
    assert abs(st.rel_res0 / (r / f) - 1.0) <= 17 * 2.0 ** -24
    s.close()
