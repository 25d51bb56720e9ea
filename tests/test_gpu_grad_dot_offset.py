"""mg_grad_dot of potentials (steep spectra: small gradients) with and without a constant, against
the same sum in extended precision: the error is that of the gradient's terms, not of u's size."""
import numpy as np
import pytest

from synth import grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EPS = 2.0 ** -52


@pytest.mark.parametrize("order", [2, 4])
@pytest.mark.parametrize("shape,offset", [((7, 5, 9), 0), ((16, 24, 40), 1), ((48, 40, 64), 0), ((32, 48, 112), 0)])
@pytest.mark.parametrize("mean", [0.0, 1e3, 1e6])
def test_a_constant_does_not_matter(gb, shape, offset, order, mean):
    rng = np.random.default_rng(13)
    w = rng.standard_normal((3,) + shape).astype(np.float32)
    u = grf(shape, 14, -6.0) + mean
    n = u.size
    s = gb.Solver(shape)
    wb = torch.empty(3 * n + offset, dtype=torch.float32, device="cuda")
    ub = torch.empty(n + offset, dtype=torch.float64, device="cuda")
    wd, ud = wb[offset:].view((3,) + shape), ub[offset:].view(shape)
    wd.copy_(torch.from_numpy(w))
    ud.copy_(torch.from_numpy(u))
    x = u.astype(np.longdouble)
    ref, bar = np.longdouble(0), 0.0
    for a in range(3):
        d1 = np.roll(x, -1, 2 - a) - np.roll(x, 1, 2 - a)
        d2 = np.roll(x, -2, 2 - a) - np.roll(x, 2, 2 - a)
        g, m = ((8 * d1 - d2) / 12, (8 * abs(d1) + abs(d2)) / 12) if order == 4 else (d1 / 2, abs(d1) / 2)
        ref += (w[a] * g).sum()
        bar += float((abs(w[a]) * m).sum())
    # two roundings per difference and product, then a chain of 3 x 2 x 16 terms per thread and
    # 10 + 10 levels of block sums, each off by half an EPS of no more than the sum of magnitudes
    got = float(s.grad_dot(ud, wd, order))
    assert abs(got - float(ref)) <= 0.5 * EPS * (4 + 96 + 20) * bar
    s.close()


@pytest.mark.parametrize("shape,offset", [((8, 12, 16), 0), ((8, 12, 16), 1)])
def test_subnormal_and_infinite_weights(gb, shape, offset):
    rng = np.random.default_rng(15)
    n = int(np.prod(shape))
    s = gb.Solver(shape)
    u = rng.standard_normal(shape)
    wb = torch.empty(3 * n + offset, dtype=torch.float32, device="cuda")
    ub = torch.empty(n + offset, dtype=torch.float64, device="cuda")
    wd, ud = wb[offset:].view((3,) + shape), ub[offset:].view(shape)
    ud.copy_(torch.from_numpy(u))
    # weights of every kind, alone and beside others: subnormal, zero, smallest and largest normal
    for pool in ([2.0 ** -149, -2.0 ** -130, 0.0, 2.0 ** -126], [3.0, -0.0, 2.0 ** -140], [2.0 ** 127, -2.0 ** -149]):
        w = rng.choice(np.array(pool, dtype=np.float32), (3,) + shape)
        wd.copy_(torch.from_numpy(w))
        for order in (2, 4):
            terms = []
            for a in range(3):
                d1 = np.roll(u, -1, 2 - a) - np.roll(u, 1, 2 - a)
                d2 = np.roll(u, -2, 2 - a) - np.roll(u, 2, 2 - a)
                terms.append(w[a].astype(np.float64) * ((8 * d1 - d2) / 12 if order == 4 else d1 / 2))
            terms = np.stack(terms)
            # n terms of both signs: half an EPS of the sum of magnitudes for each of some 100 roundings
            assert abs(float(s.grad_dot(ud, wd, order)) - terms.sum()) <= 60 * EPS * np.abs(terms).sum()
    for bad in (np.inf, np.nan):
        w = rng.standard_normal((3,) + shape).astype(np.float32)
        w[1, 2, 3, 4] = bad
        wd.copy_(torch.from_numpy(w))
        got = float(s.grad_dot(ud, wd, 4))
        assert np.isnan(got) if np.isnan(bad) else np.isinf(got)
    s.close()
