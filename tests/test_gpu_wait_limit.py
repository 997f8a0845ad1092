"""The bound on device waits covers both sweeps: with a bound of zero each gives
up before its first step and reports it as a status, through the stage that runs
it alone, and the CUDA context stays usable.  With the default bound the same
sweep, with many strips that wait for each other, finishes."""
import numpy as np
import pytest

from paper_1704_03151_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_evolution_sweep_gives_up(precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03151_gb300 import miugks
    case = wl.cavity(nx=96, ny=80, nvel=8, kn=0.5, lid=0.2, levels=1)
    rng = np.random.default_rng(3)
    it, r = rng.uniform(0.2, 3.0, 96 * 80), rng.normal(size=(2, 96 * 80, 64))
    a = miugks.Solver(case, precision=precision)
    x = a.sgs_micro(0, it, r)
    a.set_wait_limit(0.0)
    with pytest.raises(miugks.MiugksError) as e:
        a.sgs_micro(0, it, r)
    assert e.value.status == miugks.MIUGKS_ETIMEOUT
    b = miugks.Solver(case, precision=precision)
    b.set_wait_limit(0.5)
    assert np.array_equal(b.sgs_micro(0, it, r), x)
