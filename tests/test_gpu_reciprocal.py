"""rcp64 (one third-order step from a single-precision seed) against the division,
over every exponent and at the edges where it hands over to the division.

With a seed within 2^-22 of 1/x the step leaves a relative error below 2^-66 before
its one rounding, so the result is the quotient or its neighbour: one unit in the last
place.  Outside the exponents of the seed the result is the division's, bit for bit."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "common.cuh"
__global__ void k(const double* x, double* y, int n)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < n) y[t] = miugks::rcp64(x[t]);
}
extern "C" int reciprocals(const double* x, double* y, int n)
{
    k<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}
"""


def test_against_division(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import build
    src, lib = tmp_path / "rcp.cu", tmp_path / "librcp.so"
    src.write_text(SOURCE)
    subprocess.check_call([build._nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", "-o", str(lib), str(src)])
    rng = np.random.default_rng(1)
    exps = np.repeat(np.arange(-1074, 1024), 64)
    with np.errstate(over="ignore", under="ignore"):
        x = np.ldexp(1.0 + rng.random(exps.size), exps) * rng.choice([-1.0, 1.0], exps.size)
        edge = np.ldexp(1.0, np.arange(-102, 103))
        x = np.concatenate([x, edge, np.nextafter(edge, 0.0), np.nextafter(edge, np.inf), -edge,
                            [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1.7976931348623157e308]])
    d = torch.from_numpy(x).cuda()
    y = torch.empty_like(d)
    assert ctypes.CDLL(str(lib)).reciprocals(ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(y.data_ptr()), x.size) == 0
    y = y.cpu().numpy()
    with np.errstate(all="ignore"):
        q = 1.0 / x
        e = np.frexp(x)[1] - 1
        outside = ~np.isfinite(x) | (x == 0.0) | (e < -99) | (e > 99)
    assert np.array_equal(y[outside], q[outside], equal_nan=True)
    ulps = np.abs(y[~outside].view(np.int64) - q[~outside].view(np.int64))
    assert np.max(ulps) <= 1
