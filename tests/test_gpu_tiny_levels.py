"""Evolution sweep on levels of a few cells, whose lines' wall sums have as many shares as velocities: against the
oracle's serial sweep, with the bounds of test_gpu_sweep_strips.py, and no slower than on a larger level."""
import numpy as np
import pytest

import oracle
from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def box(nx, ny, nu, nv, levels=1):
    c = wl.cavity(nx=nx, ny=ny, nvel=8, lid=0.2, levels=levels)
    c["vgrid"] = dict(c["vgrid"], nu=nu, nv=nv)
    return c


def solver(case, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    return miugks.Solver(case, precision=precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nu,nv", [(3, 4), (13, 29), (47, 13), (48, 48)])
@pytest.mark.parametrize("level", [0, 1, 2])
def test_sweep_matches_serial_order(level, nu, nv, precision):
    case = box(12, 4, nu, nv, levels=3)              # levels of 12x4, 6x2 and 3x1 cells
    o, g = oracle.Oracle(case), solver(case, precision)
    rng = np.random.default_rng(6)
    nc = (12 >> level) * (4 >> level)
    it, r = rng.uniform(0.2, 3.0, nc), rng.standard_normal((2, nc, o.nv))
    x, y = g.sgs_micro(level, it, r), o.sgs_micro(level, it, r)
    assert np.max(np.abs(x - y)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(y))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_wall_sums_of_a_tiny_level_take_no_longer(precision):
    """The sums of 2x2 cells are over the same velocities as those of 16x16: their launches may take longer by the
    spread of short launches, not by a multiple."""
    import torch

    def device_time(n):
        s = solver(box(n, n, 48, 13), precision)
        s.init_uniform(1.0, 0.0, 0.0, 1.0)
        s.step(3)
        for _ in range(2):                           # (the first profile of a process may come out empty)
            with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as p:
                s.step(10)
                torch.cuda.synchronize()
        t = [e.time_range.elapsed_us() for e in p.events() if "k_line_rho" in e.name]
        if not t:
            pytest.skip("the profiler records no launches")
        return float(np.median(t))

    assert device_time(2) <= 2.0 * device_time(16)
