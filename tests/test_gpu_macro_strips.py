"""Prediction sweep (Eq. macroFinalDefect) at the sizes where its strips of grid
lines can go wrong: strips of 32 (mixed) and 8 (FP64) lines, full, one line
short and one line over, lines along either axis, one cell long, many strips,
and around a body.  Against the oracle's serial sweep.  The FP64 bound is the
parity bound of the other stages; in the mixed form a value is the end of a
chain of at most nx + ny FP32 updates whose coupling coefficients add up to less
than one, so its error stays within a few dozen FP32 roundings (2^-24 each) of
the largest value: 2e-5 covers several hundred.
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


BODY = wl.square_cylinder(ma=0.5, kn=0.5, nvel=8, vmax=5.0, levels=1, nx_side=8, nx_sq=4, ny_side=16, ny_sq=8, half=3.0,
                          dtn_growth=0.0)
CASES = [wl.cavity(nx=nx, ny=ny, nvel=6, lid=0.2, levels=1)
         for nx, ny in ((1, 9), (7, 8), (8, 7), (9, 33), (32, 31), (33, 40), (65, 64), (130, 70), (70, 130), (256, 300))]
CASES += [wl.couette(n=34, nx=17, nvel=6, t_top=1.3), BODY]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: c["name"])
def test_sweep_matches_serial_order(lib, case, precision):
    rng = np.random.default_rng(11)
    nc = case["nx"] * case["ny"]
    rho, t = rng.uniform(0.7, 1.4, nc), rng.uniform(0.8, 1.3, nc)
    u, v = rng.uniform(-0.3, 0.3, (2, nc))
    W = np.stack([rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v) + 0.75 * rho * t], axis=1)
    R = rng.normal(size=(nc, 4))
    if case.get("solid") is not None:
        R[np.asarray(case["solid"]) > 0] = 0.0
    o, g = oracle.Oracle(case), lib.Solver(case, precision=precision)
    o.init_uniform(1.0, 0.0, 0.0, 1.0)
    g.init_uniform(1.0, 0.0, 0.0, 1.0)
    x, y = g.sgs_macro(0, W, W, R), o.sgs_macro(0, W, W, R)
    assert np.max(np.abs(x - y)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(y))
