"""The bottom cycle in one CTA against the one-kernel-per-operation chain: the same bits on
bottom hierarchies with short z columns, more columns than threads (20 x 20 x 10), odd
coarsest sides, two to four levels and a coarsest level of several hundred cells."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("degree", [1, 3, 4])
@pytest.mark.parametrize("shape", [(16, 16, 16), (20, 40, 40), (10, 20, 20), (8, 20, 24), (8, 8, 64), (12, 24, 8),
                                   (64, 64, 64), (14, 10, 10)])
def test_small_cycle_equals_chain(gb, shape, degree):
    r = torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(91), device="cuda")
    a, b = gb.Solver(shape, degree=degree), gb.Solver(shape, degree=degree, fused=False)
    assert torch.equal(a.vcycle(r).view(torch.int32), b.vcycle(r).view(torch.int32))
    a.close()
    b.close()
