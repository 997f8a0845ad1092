"""Solvers of different sizes, each in a host thread of its own.

A launch asks for shared memory by its solver's mesh and velocity grid, and the
limit it has to stay under belongs to the kernel, which the threads share.  One
thread's solver needs far more than another's (lines, strips and velocities of
the flux cache), every iteration is eager (stage timing), so the launches of the
two interleave; the results have to be those of a run alone, bit for bit."""
import threading

import numpy as np
import pytest

from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_threads_with_solvers_of_different_sizes(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    miugks.load()
    cases = [wl.cavity(nx=12, ny=16, nvel=8, kn=0.5, lid=0.2, levels=1), wl.cavity(nx=96, ny=120, nvel=10, kn=0.5, lid=0.2, levels=2),
             wl.cavity(nx=8, ny=6, nvel=48, kn=0.5, lid=0.2, levels=1)]

    def run(case, out, q, n):
        try:
            s = miugks.Solver(case, stream=torch.cuda.Stream(), precision=precision)
            s.set_timing(True)
            s.init_fields(*wl.random_fields(case, q, amp=0.02))
            for _ in range(n):
                s.step(1)
            out[q] = s.get_f()
        except Exception as e:                  # reported by the main thread
            out[q] = e

    n, alone, together = 40, [None] * 3, [None] * 3
    for q, c in enumerate(cases):
        run(c, alone, q, n)
    threads = [threading.Thread(target=run, args=(c, together, q, n)) for q, c in enumerate(cases)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, together):
        assert not isinstance(a, Exception) and not isinstance(b, Exception), (a, b)
        assert np.array_equal(a, b)
