"""Two live batches whose bottom cycles need different amounts of shared memory: the limit that
the second one sets on the kernels they share does not take the first one's launches away."""
import pytest
import torch

from synth import grf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [1, 3])
def test_a_batch_with_a_smaller_bottom_leaves_the_first_alone(gb, degree):
    # 64^3: bottom cycle from 16^3 (93 KB); 96^3: from 12^3 (36 KB)
    shapes = [(64, 64, 64), (64, 64, 128)]
    F = [torch.from_numpy(grf(s, 310 + i)).cuda() for i, s in enumerate(shapes)]

    def history(batch, graph):
        batch.use_graph(graph)
        phi = [torch.zeros_like(f) for f in F]
        stats, _ = batch.solve(F, phi, tol=0.0, max_vcycles=6 if graph else 7)   # (a new key each: captured anew)
        return phi, [s.history[:6] for s in stats]

    a = gb.Batch(shapes, degree=degree)
    phi0, before = history(a, True)
    b = gb.Batch([(96, 96, 96)], degree=degree)
    # the phase graph and the persistent kernel sum the residual's squares over other tiles, so
    # the histories tell which of them ran
    _, persistent = history(a, False)
    a.solve(F, [torch.zeros_like(f) for f in F], tol=1e-3)
    a.use_graph(True)
    a.solve(F, [torch.zeros_like(f) for f in F], tol=1e-3)
    phi1, after = history(a, True)
    assert before != persistent
    assert after == before
    assert all(torch.equal(p, q) for p, q in zip(phi0, phi1))
    b.close()
    a.close()
