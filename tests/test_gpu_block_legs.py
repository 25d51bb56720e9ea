"""Block kernels of the levels between the bottom cycle and the streaming legs, and the legs'
schedules, against the one-kernel-per-operation chain (GPU): the same operations per cell, so
the corrections agree bit for bit."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# level 0 or 1 in blocks of 8^3: whole blocks; sides that end inside a block; two blocked
# levels; the largest.  Then levels whose legs run an equal number of CTAs per tile.
SHAPES = [(32, 32, 32), (16, 24, 40), (20, 36, 40), (44, 20, 36), (72, 40, 40), (40, 40, 72), (56, 56, 56),
          (80, 80, 80), (96, 96, 96), (144, 80, 80)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("degree", [1, 2, 3])
def test_block_legs_bit_identical_to_chain(gb, shape, degree):
    g = torch.Generator(device="cuda").manual_seed(31)
    r = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    a = gb.Solver(shape, prec="mixed", fused=1, degree=degree).vcycle(r)
    b = gb.Solver(shape, prec="mixed", fused=False, degree=degree).vcycle(r)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
