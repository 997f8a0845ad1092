"""Interface flux (Step 1) over the velocity grids where its thread layout and its
shared-memory cache can go wrong: columns that fill a block, are longer than one
or leave part of it idle, very short axes, nodes at zero on either axis (the
mean of both sides), grids on both sides of the cache limit, and a domain edge
with every boundary type beside it.  Against the oracle's flux.  The FP64 bound
is the parity bound of the other stages.  In the mixed form a flux is a product
of a few dozen FP32 factors and sums whose terms are of the flux's own size (the
reconstruction differences carry a factor of order one here), so a few dozen
roundings of 2^-24: 2e-5 covers several hundred.
"""
import numpy as np
import pytest

import oracle
from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    miugks.load()
    return miugks


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("nu,nv", [(6, 6), (9, 9), (8, 300), (40, 7), (33, 31), (32, 47), (48, 49), (57, 60), (89, 89)])
def test_flux_matches_oracle(lib, nu, nv, precision):
    c = wl.cavity(nx=4, ny=3, nvel=8, lid=0.2, levels=1, vmax=5.0)
    c["vgrid"] = dict(c["vgrid"], nu=nu, nv=nv)
    c["bcs"][1] = wl.bc(wl.OUTFLOW)
    c["bcs"][3] = wl.bc(wl.FARFIELD, rho=1.1, u=0.3, t=1.2)
    c["bcs"][0] = wl.bc(wl.SYMMETRY)
    o, g = oracle.Oracle(c), lib.Solver(c, precision=precision)
    o.init_fields(*wl.random_fields(c, 4, amp=0.2))
    f = o.get_f() * (1.0 + 0.05 * np.random.default_rng(9).standard_normal((2, 12, o.nv)))
    f = f.astype(np.float32).astype(np.float64)      # the same state in both forms
    o.set_f(f)
    g.set_f(f)
    for a, b in zip(g.stage_flux(), o.stage_flux()):
        assert np.max(np.abs(a - b)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(b))
