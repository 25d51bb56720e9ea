"""mg_cic_paint where its integer weights can go wrong: fractions of zero and one ulp, positions
on and beyond the mesh's ends and below 2^-8 (the FP64 form), masses of every kind."""
import numpy as np
import pytest

from oracle import pm

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def positions(rng, shape, n):
    side = np.array(shape[::-1], dtype=np.float32)
    p = (rng.random((n, 3)) * side).astype(np.float32)
    special = np.array([0.0, -0.0, 1.0, 2.0 ** -8, 2.0 ** -9, 1e-6, 1e-30, -1e-6, -2.0 ** -8, -0.5, -3.75, 7.9999995,
                        np.nextafter(np.float32(1), np.float32(0)), 8.0, 15.999999, 16.0, 100.25, -100.25, 4e6, 5e6,
                        1e9, -1e9], dtype=np.float32)
    k = len(special)
    for a in range(3):
        p[a * k:(a + 1) * k, a] = special
    return p


@pytest.mark.parametrize("shape", [(8, 8, 8), (8, 16, 24), (5, 7, 9)])
@pytest.mark.parametrize("mass", [1.0, 0.37, -2.5, 0.0, 1e-280, 1e-310, 1e290, "array"])
def test_paint_weights(gb, shape, mass):
    rng = np.random.default_rng(98)
    p = positions(rng, shape, 400)
    m = mass
    if mass == "array":
        m = rng.standard_normal(400).astype(np.float32)
        m[:4] = [0.0, 1e-40, 1.0, -1.0]
    s = gb.Solver(shape)
    mt = torch.from_numpy(m).cuda() if mass == "array" else mass
    got = s.cic_paint(torch.from_numpy(p).cuda(), mt).cpu().numpy()
    md = m.astype(np.float64) if mass == "array" else m
    ref = pm.cic_paint(p, md, shape)
    # three roundings per contribution in the oracle and one here, and at most 400 sums on
    # either side
    scale = pm.cic_paint(p, np.abs(md) if mass == "array" else abs(mass), shape)
    assert np.all(np.abs(got - ref) <= 804 * 2.0 ** -53 * scale + 400 * 5e-324)
    s.close()
