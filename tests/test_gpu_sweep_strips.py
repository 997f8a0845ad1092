"""Evolution sweep (Eq. microFinalDefect) at the sizes where its strips of grid
lines and runs of velocities can go wrong: one line, strips full, one short and
one over for 8, 16 and 32 lines per strip, lines along either axis, more lines
than 128 and 256 (fewer lanes per cell), velocity counts around the padding of a
row and around the 128 leaving velocities of one block of the line walk, every
boundary type at an edge, and a body.  Against the oracle's serial sweep.  The
FP64 bound is the parity bound of the other stages; in the mixed form a value is
the end of a chain of contractions (each cell's coefficients sum to less than
one), so its error stays within a few dozen FP32 roundings of the largest value:
2e-5 covers several hundred.
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


def grid(case, nu, nv):
    case["vgrid"] = dict(case["vgrid"], nu=nu, nv=nv)
    case["name"] += "_%dx%d" % (nu, nv)
    return case


def edges(nx, ny, types):
    """A box whose west, east, south and north edges have the given boundary types."""
    c = wl.cavity(nx=nx, ny=ny, nvel=8, lid=0.2, levels=1)
    for b, t in zip((3, 1, 0, 2), types):
        c["bcs"][b] = wl.bc(t, u=0.1, t=1.2)
    c["name"] += "_%d%d%d%d" % tuple(types)
    return c


W, S, F, O = wl.WALL, wl.SYMMETRY, wl.FARFIELD, wl.OUTFLOW
CASES = [grid(wl.cavity(nx=nx, ny=ny, nvel=8, lid=0.2, levels=1), nu, nv)
         for nx, ny, nu, nv in ((1, 9, 3, 5), (7, 8, 16, 17), (8, 9, 15, 17), (17, 16, 16, 16), (33, 31, 9, 9), (65, 24, 12, 12),
                                (12, 129, 48, 47), (130, 140, 6, 6), (257, 260, 4, 4), (300, 20, 5, 7), (40, 40, 48, 46))]
CASES += [edges(9, 12, t) for t in ((W, S, F, O), (S, S, W, W), (O, W, W, O), (S, W, S, F), (S, O, O, S))]
CASES += [grid(wl.square_cylinder(ma=0.5, kn=0.5, nvel=8, vmax=5.0, levels=1, nx_side=8, nx_sq=4, ny_side=16, ny_sq=8, half=3.0,
                                  dtn_growth=0.0), 17, 16)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: c["name"])
def test_sweep_matches_serial_order(lib, case, precision):
    o, g = oracle.Oracle(case), lib.Solver(case, precision=precision)
    rng = np.random.default_rng(5)
    nc = case["nx"] * case["ny"]
    it, r = rng.uniform(0.2, 3.0, nc), rng.normal(size=(2, nc, o.nv))
    if case.get("solid") is not None:
        r[:, np.asarray(case["solid"]) > 0] = 0.0
    y = o.sgs_micro(0, it, r)
    for _ in range(2):                      # the second sweep starts from the first one's values in x
        x = g.sgs_micro(0, it, r)
        assert np.max(np.abs(x - y)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(y))
