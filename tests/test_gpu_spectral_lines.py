"""The spectral scheme's transforms by line: short powers of two (4 points per thread), long ones (16),
one axis in registers beside a mixed-radix one, passes large enough for the L2 prefetch, and
single precision with strong linear growth (its own transforms).  Bounds as in
test_gpu_spectral.py: FP64 1e-12 of the field scale, FP32 relative L2 1e-5, against numpy."""
import numpy as np
import pytest

from oracle import spectral as SO

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


def check(sp, model, shape, dtype, dt, n, **kw):
    with sp.Simulation(model, shape, dt=dt, dtype=dtype, scheme=sp.SCHEME_SPECTRAL, seed=31, **kw) as s:
        u0 = s.read(0)
        s.step(n)
        got = s.read(0)
    ref = SO.step(model, u0, dt=dt, nsteps=n)
    if dtype == 0:
        assert np.abs(got - ref).max() <= 1e-12 * max(1.0, np.abs(ref).max())
    else:
        assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("model,shape", [(1, (32, 32)), (0, (64, 32)), (1, (1024, 64)), (1, (48, 256)), (0, (256, 48)),
                                         (1, (2048, 35)), (1, (63, 2048)), (0, (32, 32, 32)), (1, (40, 64, 32)),
                                         (0, (64, 30, 128)), (1, (32, 128, 21)), (1, (2048, 4096))])
def test_lines(sp, model, shape, dtype):
    check(sp, model, shape, dtype, 0.1, 4 if np.prod(shape) > 1 << 20 else 12, ic_amp=0.4)


@pytest.mark.parametrize("model,dt,amp", [(0, 0.5, 0.4), (0, 0.3, 0.4), (1, 1.2, 0.05)])
@pytest.mark.parametrize("shape", [(64, 128), (96, 40), (35, 63), (32, 16, 64), (12, 20, 30)])
def test_strong_linear_growth_in_single_precision(sp, shape, model, dt, amp):
    """1 / (1 - dt max L) of 2, 1.43 and 1.43."""
    check(sp, model, shape, 1, dt, 10, ic_amp=amp)
