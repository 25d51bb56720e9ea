"""mg_grad (transposed) and mg_grad_dot against FP64 numpy at the edges of their paths: pairs
and odd rows, misaligned views, z chunks with a remainder, cells that leave the FP32 range."""
import numpy as np
import pytest

from oracle import grad

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EPS = 2.0 ** -52


def oracle(order):
    return (grad.grad4_T, grad.grad4) if order == 4 else (grad.grad2_T, grad.grad2)


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("shape,offset", [((4, 4, 4), 0), ((7, 5, 9), 0), ((16, 24, 40), 0), ((16, 24, 40), 1),
                                          ((80, 96, 64), 0), ((160, 160, 128), 0)])
def test_grad_transpose_and_dot(gb, shape, offset, order):
    rng = np.random.default_rng(11)
    n = int(np.prod(shape))
    w = rng.standard_normal((3,) + shape).astype(np.float32)
    u = rng.standard_normal(shape)
    s = gb.Solver(shape)
    wb = torch.empty(3 * n + offset, dtype=torch.float32, device="cuda")
    ub = torch.empty(n + offset, dtype=torch.float64, device="cuda")
    wd, ud = wb[offset:].view((3,) + shape), ub[offset:].view(shape)
    wd.copy_(torch.from_numpy(w))
    ud.copy_(torch.from_numpy(u))
    gT, g = oracle(order)
    ref = gT(w.astype(np.float64))
    # a cell sums 12 (6) terms of size <= 8 max|w| / 12 in FP64: a few roundings of that size
    bar = 12 * EPS * np.abs(w).max()
    assert np.abs(s.grad_T(wd, order).cpu().numpy() - ref).max() <= bar
    dot = float((u * ref).sum())
    assert abs(float(s.grad_dot(ud, wd, order)) - dot) <= 8 * EPS * np.abs(u * ref).sum() + bar * np.abs(u).sum()
    s.close()


@pytest.mark.parametrize("scale", [0.0, 2.0 ** -120, 2.0 ** -60, 2.0 ** 100, 2.0 ** 126])
def test_grad_transpose_outside_the_expansion_range(gb, scale):
    shape = (8, 8, 8)
    rng = np.random.default_rng(12)
    w = (rng.uniform(-1, 1, (3,) + shape) * scale).astype(np.float32)
    w[0, 3, 3, 3] = 1.0  # one cell of ordinary size among them
    s = gb.Solver(shape)
    ref = grad.grad4_T(w.astype(np.float64))
    out = s.grad_T(torch.from_numpy(w).cuda(), 4).cpu().numpy()
    assert np.abs(out - ref).max() <= 12 * EPS * np.abs(w).max()
    w[1, 2, 2, 2] = np.inf
    w[2, 5, 5, 5] = np.nan
    ref = grad.grad4_T(w.astype(np.float64))
    out = s.grad_T(torch.from_numpy(w).cuda(), 4).cpu().numpy()
    assert np.array_equal(np.isfinite(out), np.isfinite(ref))
    assert np.array_equal(np.isnan(out), np.isnan(ref))
    s.close()
