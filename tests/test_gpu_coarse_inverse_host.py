"""The coarsest inverse where the GPU refuses the kernel's resident grid (here on request): the
host forms it, with the same bits and the same refusals."""
import numpy as np
import pytest

from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape,levels", [((4, 5, 6), 1), ((8, 8, 8), 1), ((20, 40, 24), 0)])
def test_host_inverse_has_the_kernels_bits(gb, shape, levels, sym):
    psi = torch.from_numpy(smoothed_grf(shape, 100, 1.0, 0.4)).cuda()
    gpu, host = (gb.Solver(shape, op="curv", levels=levels, curv_sym=sym) for _ in range(2))
    gb._check(gb.lib().mg_set_cycle_graphs(host._c(), gb.TEST_REFUSE))
    F = torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(101), device="cuda", dtype=torch.float64)
    r = torch.randn(gpu.level_shape(gpu.levels - 1), generator=torch.Generator(device="cuda").manual_seed(102),
                    device="cuda", dtype=torch.float64)
    got = []
    for s in (gpu, host):
        s.set_geometry(psi)
        phi, st = s.solve(F, tol=1e-6, max_vcycles=100)
        bar, _, sa = s.solve_adjoint(F, tol=1e-6, max_vcycles=100)   # (the transposed inverse)
        got.append((s.coarse_solve(r), phi, bar))
    assert all(torch.equal(a, b) for a, b in zip(*got))
    # a folded mesh is refused by either, and both are usable afterwards
    z = np.arange(float(shape[0]))
    fold = 40.0 * np.cos(2 * np.pi * z / shape[0])[:, None, None] + np.zeros(shape)
    for s in (gpu, host):
        with pytest.raises(gb.GbmgError) as e:
            s.set_geometry(torch.from_numpy(fold).cuda())
        assert e.value.status == 1
        s.set_geometry(psi)
        assert torch.equal(s.coarse_solve(r), got[0][0])
        s.close()
