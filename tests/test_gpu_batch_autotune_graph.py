"""The autotuner of a batch that the phase graph serves: it tunes what that graph reads (the
level-0 tile size) and leaves the persistent kernel's grid and other tile sizes alone."""
import pytest
import torch

from synth import grf

pytestmark = pytest.mark.gpu


def test_autotune_keeps_what_the_phase_graph_does_not_read(gb):
    shapes = [(64, 64, 64)] * 3 + [(96, 96, 96), (128, 128, 128)]
    F = [torch.from_numpy(grf(s, 330 + i)).cuda() for i, s in enumerate(shapes)]
    batch = gb.Batch(shapes)
    batch.use_graph(True)
    ref = [torch.zeros_like(f) for f in F]
    batch.solve(F, ref, tol=1e-8)
    tiles = batch.tiles()
    batch.set_blocks(61)
    phi = [torch.zeros_like(f) for f in F]
    blocks, tuned = batch.autotune(F, phi, tol=1e-8)
    assert blocks == 61 and tuned[1:] == tiles[1:]
    assert batch.tiles() == tuned
    for p, r in zip(phi, ref):   # (the level-0 tiles sum the means in another order)
        assert (p - r).norm() <= 1e-7 * r.norm()
    batch.close()
