"""Prediction sweep of the mixed form where a ring of eight steps no longer fits
beside the edge values: more than 224 grid lines of more than 396 cells along x.
One size on either side of that line and the largest mesh, against the oracle's
serial sweep with the bound of test_gpu_macro_strips.py."""
import numpy as np
import pytest

import oracle
from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(396, 225), (397, 225), (512, 256)])
def test_sweep_matches_serial_order(nx, ny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    c = wl.cavity(nx=nx, ny=ny, nvel=4, lid=0.2, levels=1)
    rng = np.random.default_rng(11)
    n = nx * ny
    rho, t = rng.uniform(0.7, 1.4, n), rng.uniform(0.8, 1.3, n)
    u, v = rng.uniform(-0.3, 0.3, (2, n))
    w = np.stack([rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v) + 0.75 * rho * t], axis=1)
    r = rng.normal(size=(n, 4))
    o, g = oracle.Oracle(c), miugks.Solver(c, precision="mixed")
    o.init_uniform(1.0, 0.0, 0.0, 1.0)
    g.init_uniform(1.0, 0.0, 0.0, 1.0)
    x, y = g.sgs_macro(0, w, w, r), o.sgs_macro(0, w, w, r)
    assert np.max(np.abs(x - y)) <= 2e-5 * np.max(np.abs(y))
