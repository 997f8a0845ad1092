"""Interface flux at the ends of its values' range.

A NaN in one cell reaches the cells that share a face with it and no others: the
limiter gives a face beyond them no slope, as the oracle's does (the iteration
then reports divergence instead of spreading it).  And in FP64 densities far
outside FP32's range are ordinary numbers.  Bounds as for the other fluxes."""
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


def state(lib, precision):
    c = wl.cavity(nx=8, ny=6, nvel=8, lid=0.2, levels=1)
    o, g = oracle.Oracle(c), lib.Solver(c, precision=precision)
    o.init_fields(*wl.random_fields(c, 4, amp=0.2))
    return o, g, o.get_f().astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_nan_stays_beside_its_cell(lib, precision):
    o, g, f = state(lib, precision)
    f[0, 20, :] = np.nan
    o.set_f(f)
    g.set_f(f)
    for a, b in zip(g.stage_flux(), o.stage_flux()):
        ok = np.isfinite(b)
        assert not np.all(ok) and np.array_equal(np.isfinite(a), ok)
        assert np.max(np.abs(a[ok] - b[ok])) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(b[ok]))


@pytest.mark.parametrize("scale", [1e-100, 1e-60, 1e-20, 1e20, 1e60])
def test_densities_outside_single_precision(lib, scale):
    o, g, f = state(lib, "fp64")
    o.set_f(f * scale)
    g.set_f(f * scale)
    for a, b in zip(g.stage_flux(), o.stage_flux()):
        assert np.all(np.isfinite(a))
        assert np.max(np.abs(a - b)) <= 1e-10 * np.max(np.abs(b))
