"""Velocity grids with a very long first axis.

The FP64 flux keeps constants per node of that axis in shared memory, which end
at about 2,200 nodes; beyond it forms them where they are used.  One node count
on either side of that line, and one that only the mixed form's smaller tables
ever had room for, against the oracle's flux, and an iteration after it.  The
bounds are those of the flux on shorter axes: each velocity's arithmetic is the
same, and the sums' rounding grows with the root of the count at most."""
import numpy as np
import pytest

import oracle
from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,nu", [("fp64", 2150), ("fp64", 2401), ("fp64", 4801), ("mixed", 4801)])
def test_flux_and_iteration(precision, nu):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    c = wl.cavity(nx=3, ny=2, nvel=8, lid=0.2, levels=1, vmax=5.0)
    c["vgrid"] = dict(c["vgrid"], nu=nu, nv=3)
    o, g = oracle.Oracle(c), miugks.Solver(c, precision=precision)
    o.init_fields(*wl.random_fields(c, 4, amp=0.2))
    f = o.get_f() * (1.0 + 0.05 * np.random.default_rng(9).standard_normal((2, 6, o.nv)))
    f = f.astype(np.float32).astype(np.float64)
    for s in (o, g):
        s.set_f(f)
    tol = 1e-10 if precision == "fp64" else 2e-5
    for a, b in zip(g.stage_flux(), o.stage_flux()):
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b))
    r = o.step(1)
    assert np.max(np.abs(g.step(1) - r)) <= tol * np.max(r)
