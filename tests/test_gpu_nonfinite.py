"""Non-finite values in the sweeps stop at bodies.

An overflow ahead of a strong shock is an ordinary event of a Mach 5 start: the
cell where it ends keeps its state, and a body, whose cells have no equation,
must come out of every sweep with exact zeros and shield what lies behind it.
An infinity planted ahead of a body must reach the cells that it reaches in the
oracle's serial sweep and no others, and the values elsewhere must be the
oracle's (the parity bounds of the sweeps' other tests).
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


def body(wide):
    """A body in a stream, its faces open, so that a velocity is not coupled to others."""
    n = dict(nx_side=16, nx_sq=8, ny_side=8, ny_sq=4) if wide else dict(nx_side=8, nx_sq=4, ny_side=16, ny_sq=8)
    c = wl.square_cylinder(ma=0.5, kn=0.5, nvel=8, vmax=5.0, levels=1, half=3.0, dtn_growth=0.0, **n)
    c["bcs"] = [wl.bc(wl.FARFIELD, u=0.1) for _ in c["bcs"]]
    return c


def agrees(x, y, tol):
    ok = np.isfinite(y)
    assert np.array_equal(np.isfinite(x), ok)
    assert np.max(np.abs(x[ok] - y[ok])) <= tol * np.max(np.abs(y[ok]))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("wide", [False, True])
def test_prediction_sweep(lib, wide, precision):
    c = body(wide)
    nx, n = c["nx"], c["nx"] * c["ny"]
    solid = np.asarray(c["solid"]).reshape(c["ny"], nx) > 0
    j, i = np.argwhere(solid)[0]
    rng = np.random.default_rng(11)
    rho, t = rng.uniform(0.7, 1.4, n), rng.uniform(0.8, 1.3, n)
    u, v = rng.uniform(-0.3, 0.3, (2, n))
    w = np.stack([rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v) + 0.75 * rho * t], axis=1)
    r = rng.normal(size=(n, 4))
    r[solid.ravel()] = 0.0
    r[j * nx + i - 2, 1] = np.inf
    o, g = oracle.Oracle(c), lib.Solver(c, precision=precision)
    o.init_uniform(1.0, 0.0, 0.0, 1.0)
    g.init_uniform(1.0, 0.0, 0.0, 1.0)
    x, y = g.sgs_macro(0, w, w, r), o.sgs_macro(0, w, w, r)
    assert np.all(x[solid.ravel()] == 0.0) and not np.all(np.isfinite(y))
    agrees(x, y, 1e-10 if precision == "fp64" else 2e-5)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("wide", [False, True])
def test_evolution_sweep(lib, wide, precision):
    """(Here the oracle multiplies by the zero coefficient of a downwind neighbour, so that an infinity goes
    further in it; the GPU's values beyond are held to be finite, not to be the oracle's.)"""
    c = body(wide)
    nx, n = c["nx"], c["nx"] * c["ny"]
    solid = np.asarray(c["solid"]).reshape(c["ny"], nx) > 0
    j, i = np.argwhere(solid)[0]
    o, g = oracle.Oracle(c), lib.Solver(c, precision=precision)
    rng = np.random.default_rng(5)
    it, r = rng.uniform(0.2, 3.0, n), rng.normal(size=(2, n, o.nv))
    r[:, solid.ravel()] = 0.0
    r[:, j * nx + i - 2, ::3] = np.inf
    x, y = g.sgs_micro(0, it, r), o.sgs_micro(0, it, r)
    assert np.all(x[:, solid.ravel()] == 0.0)
    ok = np.isfinite(y)
    assert not np.all(ok) and np.all(np.isfinite(x[ok]))
    tol = 1e-10 if precision == "fp64" else 2e-5
    assert np.max(np.abs(x[ok] - y[ok])) <= tol * np.max(np.abs(y[ok]))
