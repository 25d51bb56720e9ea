"""Geometries set by several host threads at once, each on its own stream, with coarsest levels
of different sizes: every call succeeds and gives the inverse of a call alone."""
import threading

import pytest

from synth import smoothed_grf

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_two_threads_invert_different_sizes(gb):
    shapes, rounds = [(4, 4, 4), (8, 8, 8)], [15000, 900]
    work = []
    for shape in shapes:
        s = gb.Solver(shape, op="curv", levels=1)
        psi = torch.from_numpy(smoothed_grf(shape, 98, 1.0, 0.4)).cuda()
        r = torch.randn(shape, generator=torch.Generator(device="cuda").manual_seed(99), device="cuda",
                        dtype=torch.float64)
        s.set_geometry(psi)
        work.append((s, psi, r, s.coarse_solve(r)))
    torch.cuda.synchronize()
    errors = []

    def run(k):
        s, psi, r, ref = work[k]
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(rounds[k]):
                    s.set_geometry(psi)
                assert torch.equal(s.coarse_solve(r), ref)
        except BaseException as e:   # (a thread's exception does not reach the test by itself)
            errors.append(e)
    threads = [threading.Thread(target=run, args=(k,)) for k in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for s, *_ in work:
        s.close()
