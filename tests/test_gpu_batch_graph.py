"""Batched solves as a graph of phase kernels against the persistent kernel (GPU): both apply
the same operations to every cell, so the iterates agree bit for bit.  The residual norms sum
the same squares over other tiles, a thread's share (up to 32 planes of four cells) in FP32:
at most 128 x 2^-24 = 8e-6 of a sum of squares on each side, 1e-5 on the ratio's root."""
import pytest
import torch

from synth import grf

pytestmark = pytest.mark.gpu

CASES = [
    # one problem; tiles of 64 x 24..32 and 32 x 32 cut in x and y; 8, 16 and 32 planes per item
    ([(32, 32, 32)], 3),
    ([(40, 72, 40), (72, 40, 56), (96, 48, 32)], 3),
    ([(64, 64, 64), (96, 96, 96), (32, 32, 32)] * 3, 3),
    ([(128, 96, 128)] * 4, 3),
    ([(72, 40, 40), (64, 64, 64)], 1),
    ([(72, 40, 40), (64, 64, 64)], 2),
    ([(72, 40, 40), (64, 64, 64)], 4),
    # no bottom cycle, levels run per operation: the persistent kernel on both sides
    ([(16, 16, 10), (48, 48, 48)], 3),
]


@pytest.mark.parametrize("shapes, degree", CASES)
def test_batch_graph_matches_persistent_kernel(gb, shapes, degree):
    F = [torch.from_numpy(grf(s, 300 + i)).cuda() for i, s in enumerate(shapes)]
    F[0] = F[0] * 1e-3                                   # scale and mean differ between problems
    F[-1] = F[-1] + 2.0
    batch = gb.Batch(shapes, degree=degree)
    ref = [torch.zeros_like(f) for f in F]
    # a guess already converged for the last problem: inactive from the first cycle
    batch.solve(F, ref, tol=1e-9, max_vcycles=40)
    start = [torch.zeros_like(f) for f in F[:-1]] + [ref[-1].clone()]
    got = {}
    for graph in (False, True):
        batch.use_graph(graph)
        for tol, maxv in ((1e-8, 40), (0.0, 2)):
            phis = [s.clone() for s in start]
            stats, _ = batch.solve(F, phis, tol=tol, max_vcycles=maxv)
            got[graph, tol] = phis, stats
    for tol in (1e-8, 0.0):
        (pa, sa), (pb, sb) = got[False, tol], got[True, tol]
        for a, b, x, y in zip(pa, pb, sa, sb):
            assert x.cycles == y.cycles and x.status == y.status
            assert torch.equal(a, b)
            assert abs(x.rel_res - y.rel_res) <= 1e-5 * x.rel_res
    batch.close()
