"""Evolution sweep with one, two and four lanes per cell, with and without
bodies, and with four steps in flight instead of eight: sizes on both sides of
the lines where launch_micro_sgs chooses (256 and 128 grid lines; runs of
velocities; 120 lines with four lanes).  Against the oracle's serial sweep, with
the bounds of test_gpu_sweep_strips.py."""
import numpy as np
import pytest

import oracle
from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def body(nx_side, nx_sq, ny_side, ny_sq, nu, nv):
    c = wl.square_cylinder(ma=0.5, kn=0.5, nvel=8, vmax=5.0, levels=1, nx_side=nx_side, nx_sq=nx_sq, ny_side=ny_side,
                           ny_sq=ny_sq, half=3.0, dtn_growth=0.0)
    c["vgrid"] = dict(c["vgrid"], nu=nu, nv=nv)
    return c


def box(nx, ny, nu, nv):
    c = wl.cavity(nx=nx, ny=ny, nvel=8, lid=0.2, levels=1)
    c["vgrid"] = dict(c["vgrid"], nu=nu, nv=nv)
    return c


CASES = {
    "one_lane_body_fp64": (body(110, 44, 108, 44, 3, 4), "fp64"),
    "two_lanes_body_mixed": (body(60, 20, 56, 24, 5, 5), "mixed"), "two_lanes_body_fp64": (body(56, 24, 60, 20, 5, 5), "fp64"),
    "four_lanes_body_fp64": (body(8, 4, 10, 4, 33, 32), "fp64"), "four_lanes_body_mixed": (body(10, 4, 8, 4, 46, 45), "mixed"),
    "four_lanes_short_ring_fp64": (box(122, 126, 33, 32), "fp64"), "four_lanes_short_ring_mixed": (box(126, 121, 46, 45), "mixed"),
    "four_lanes_long_ring_mixed": (box(30, 120, 46, 45), "mixed"),
}


@pytest.mark.parametrize("name", list(CASES))
def test_sweep_matches_serial_order(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    case, precision = CASES[name]
    o, g = oracle.Oracle(case), miugks.Solver(case, precision=precision)
    rng = np.random.default_rng(5)
    nc = case["nx"] * case["ny"]
    it, r = rng.uniform(0.2, 3.0, nc), rng.standard_normal((2, nc, o.nv))
    if case.get("solid") is not None:
        r[:, np.asarray(case["solid"]).ravel() > 0] = 0.0
    x, y = g.sgs_micro(0, it, r), o.sgs_micro(0, it, r)
    assert np.max(np.abs(x - y)) <= (1e-10 if precision == "fp64" else 2e-5) * np.max(np.abs(y))
