"""The z-marching curvilinear kernels against the one-cell tiles they replace, which still
run fields that do not start on 16 bytes: the same bits for every operator form, sweep and
residual, on meshes whose sides leave partial tiles in x (32) and y (16) and whose z runs
end on every remainder."""
import pytest

from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [False, True])
@pytest.mark.parametrize("shape", [(48, 40, 56), (80, 64, 40), (32, 40, 96), (40, 96, 64), (112, 32, 32)])
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
