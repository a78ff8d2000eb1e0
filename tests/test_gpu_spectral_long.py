"""Long runs of the spectral scheme at dt = 0.5.  The resident half spectrum's planes kx = 0 and,
for even nx, kx = nx / 2 hold both modes of conjugate pairs; their non-Hermitian part, which only
rounding makes and nothing damps, grows by up to 2 (Allen-Cahn) or 8/7 (Cahn-Hilliard) per step
unless the planes are kept Hermitian.

Reference: the oracle, restarted from its real field every 5 steps (a new transform of a real
field is Hermitian), in FP64.  Tolerance (relative L2): ten times the error of a NumPy run of
the scheme in FP32 with Hermitian planes, from the same field; u / u32 of that in FP64, but not
below 1e-12.  (That run is 1e-5 to 5e-5 off after 600 steps on these shapes where nothing but
rounding happens; where domains merge on the way the equation itself amplifies a disturbance:
64 x 96 Cahn-Hilliard from seed 31 by 2000, and 3e-3.)"""
import numpy as np
import pytest
import scipy.fft as F

from oracle import spectral as SO

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


SHAPES = [(64, 96), (45, 63), (24, 20, 30), (32, 32, 64)]


def run(sp, model, shape, dtype, n=600, chunk=100):
    with sp.Simulation(model, shape, dt=0.5, dtype=dtype, scheme=sp.SCHEME_SPECTRAL, seed=31, ic_amp=0.4) as s:
        u0 = s.read(0)
        for _ in range(n // chunk):
            s.step(chunk)
        return u0, s.read(0)


def numpy_fp32(model, u, dt, n):
    """The scheme in single precision, its two planes made Hermitian before every step."""
    shape, u = u.shape, u.astype(np.float32)
    k2 = SO.k_squared(shape, 1.0)
    den = (1.0 / (1.0 - dt * SO.linear_symbol(model, k2, 1.0, 1.0))).astype(np.float32)
    w = np.asarray(-dt if model == SO.AC else -dt * k2, dtype=np.float32)
    uh = F.rfftn(u)
    for _ in range(n):
        for kx in {0, shape[-1] // 2} if shape[-1] % 2 == 0 else {0}:
            p = uh[..., kx]
            q = np.conj(p)
            for a in range(p.ndim):
                q = np.roll(np.flip(q, a), 1, a)
            uh[..., kx] = (p + q) * np.float32(0.5)
        uh = (uh + w * F.rfftn(u * u * u)) * den
        u = F.irfftn(uh, s=shape)
    assert u.dtype == np.float32
    return u


@pytest.mark.parametrize("model,dtype", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("shape", SHAPES)
def test_long_runs_stay_with_the_oracle(sp, model, dtype, shape):
    u0, got = run(sp, model, shape, dtype)
    ref = u0
    for _ in range(120):
        ref = SO.step(model, ref, dt=0.5, nsteps=5)
    assert np.isfinite(got).all()
    tol = 10 * np.linalg.norm(numpy_fp32(model, u0, 0.5, 600) - ref)
    if dtype == 0:
        tol = max(tol * 2.0 ** -29, 1e-12 * np.linalg.norm(ref))
    assert np.linalg.norm(got - ref) <= tol


@pytest.mark.parametrize("shape", SHAPES)
def test_long_fp32_runs_with_strong_growth_stay_bounded(sp, shape):
    """FP32 with G > 4/3 keeps the rounding of its first 50 / log2 G steps; the field of the
    long run is still one of the scheme's, within |phi| = 1 and the share of 1e-2 that they add."""
    _, got = run(sp, 0, shape, 1)
    assert np.isfinite(got).all() and np.abs(got).max() < 1.02
