"""The z-marching curvilinear kernels against the one-cell tiles they replace, which still
run fields that do not start on 16 bytes: the same bits for every operator form, sweep and
residual, on meshes whose sides leave partial tiles in x (32) and y (16) and whose z runs
end on every remainder."""
import pytest

from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape", [(48, 40, 56), (80, 64, 40), (32, 40, 96), (40, 96, 64), (112, 32, 32),
                                   (64, 64, 80), (80, 112, 64), (64, 96, 112)])
def test_march_equals_tiles(gb, shape, sym):
    s = gb.Solver(shape, op="curv", curv_sym=sym)
    s.set_geometry(torch.from_numpy(smoothed_grf(shape, 81, 2.0, 0.5)).cuda())
    n = shape[0] * shape[1] * shape[2]
    g = torch.Generator(device="cuda").manual_seed(82)
    e = torch.randn(n, generator=g, device="cuda").view(shape)
    r = torch.randn(n, generator=g, device="cuda").view(shape)
    off = torch.empty(n + 1, device="cuda")[1:].view(shape)   # 4 bytes off
    off.copy_(e)
    for tr in (False, True):
        for f in (lambda u: s.curv_smooth(0, u, r, transpose=tr), lambda u: s.curv_residual(0, r, u, transpose=tr)):
            a, b = f(e), f(off)
            assert torch.isfinite(a).all() and torch.equal(a.view(torch.int32), b.view(torch.int32))
    s.close()



def turn(a, k):
    """Axes rotated: the value at (x, y, z) goes to (z, x, y) k times."""
    for _ in range(k):
        a = a.permute(1, 2, 0)
    return a.contiguous()


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape", [(16, 24, 20), (24, 40, 16), (16, 16, 14), (36, 32, 28)])
def test_step_against_turned_mesh(gb, shape, sym):
    # single-cycle residuals of the double-float step on a mesh and on the two meshes with
    # its axes turned: other tiles, runs and partial columns for the same numbers.  The
    # operator is equivariant, so the reported residuals agree to the rounding of their sums
    # and of the FP32 cycle (1e-5 of the residual before it)
    psi = torch.from_numpy(smoothed_grf(shape, 83, 2.0, 0.4)).cuda()
    F = torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(84), device="cuda",
                    dtype=torch.float64)
    seen = []
    for k in range(3):
        p, f = turn(psi, k), turn(F, k)
        s = gb.Solver(tuple(p.shape), op="curv", curv_sym=sym)
        phi, st = s.solve(f, tol=0.0, max_vcycles=3, psi=p)
        bar, _, sa = s.solve_adjoint(f, tol=0.0, max_vcycles=3)
        seen.append((st.rel_res, sa.rel_res, turn(phi, (3 - k) % 3), turn(bar, (3 - k) % 3)))
        s.close()
    for r, a, phi, bar in seen[1:]:
        assert abs(r - seen[0][0]) <= 1e-5 * seen[0][0] and abs(a - seen[0][1]) <= 1e-5 * seen[0][1]
        assert (phi - seen[0][2]).norm() <= 1e-6 * phi.norm() and (bar - seen[0][3]).norm() <= 1e-6 * bar.norm()
