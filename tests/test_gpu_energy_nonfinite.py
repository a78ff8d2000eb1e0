"""The free energy of fields with infinities, NaN or values whose fourth power overflows: what
the sum of the point densities is in FP64 arithmetic, each in the order of its terms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


def densities(q, h, c1, c2, c3, model, sp):
    p = q[0]
    g2 = 0.0
    for ax in range(p.ndim - 1, -1, -1):  # x first
        d = (np.roll(p, -1, ax) - p) / h
        g2 = g2 + d * d
    p2 = p * p
    e = 0.5 * g2 - 0.5 * c1 * p2 + 0.25 * c2 * p2 * p2
    if model == sp.MODEL_C:
        return e + 0.5 * q[1] * q[1] - c3 * p2 * q[1]
    if model == sp.MODEL_H:
        return e + 0.5 * sum(j * j for j in q[1:])
    return e


I, N = np.inf, np.nan
# model, c1, c3, field that holds the value, the value, the order parameter there (None: as it is), dtypes
CASES = [(0, 1.0, 0.5, 0, I, None, (0, 1)), (0, -1.0, 0.5, 0, I, None, (0, 1)), (0, -1.0, 0.5, 0, -I, None, (0, 1)),
         (1, -1.0, 0.5, 0, I, None, (0, 1)), (0, -1.0, 0.5, 0, N, None, (0, 1)), (0, 1.0, 0.5, 0, 1e60, None, (0,)),
         (0, 1.0, 0.5, 0, 1e100, None, (0,)), (0, 1.0, 0.5, 0, 1e200, None, (0,)), (0, 1.0, 0.5, 0, 3e38, None, (1,)),
         (3, 1.0, 0.5, 1, I, 0.5, (0, 1)), (3, 1.0, -0.5, 1, I, 0.5, (0, 1)), (3, 1.0, 0.5, 1, -I, 0.5, (0, 1)),
         (3, 1.0, 0.5, 1, I, 0.0, (0, 1)), (4, 1.0, 0.5, 1, I, None, (0, 1)), (4, 1.0, 0.5, 2, N, None, (0, 1))]


@pytest.mark.parametrize("shape", [(9, 16), (9, 13), (5, 6, 8), (3, 5, 7)])
@pytest.mark.parametrize("model,c1,c3,field,value,phi,dtypes", CASES)
def test_nonfinite_and_huge(sp, model, c1, c3, field, value, phi, dtypes, shape):
    for dtype in dtypes:
        with sp.Simulation(model, shape, dt=1e-4, dtype=dtype, c1=c1, c3=c3, ic_amp=0.5, seed=4) as sim:
            v = sim.read(field)
            at = v.size // 2
            v.ravel()[at] = value
            sim.write(field, v)
            if phi is not None:
                p = sim.read(0)
                p.ravel()[at] = phi
                sim.write(0, p)
            with np.errstate(all="ignore"):
                ref = densities([sim.read(f) for f in range(sim.nfields)], 1.0, c1, 1.0, c3, model, sp).sum()
            got = sim.reduce(sp.FREE_ENERGY)
        if np.isfinite(ref):
            assert abs(got - ref) <= 1e-14 * abs(ref), (dtype, got, ref)  # one value is all of it
        else:
            assert got == ref or (np.isnan(got) and np.isnan(ref)), (dtype, got, ref)


@pytest.mark.parametrize("h,c1,dt", [(1.0, 1e40, 1e-41), (1e-40, 1.0, 1e-82)])
@pytest.mark.parametrize("shape", [(9, 16), (5, 6, 8)])
def test_coefficients_and_steps_beyond_the_sums(sp, h, c1, dt, shape):
    for dtype in (0, 1):
        with sp.Simulation(0, shape, h=h, dt=dt, dtype=dtype, c1=c1, ic_amp=0.5, seed=4) as sim:
            q = [sim.read(0)]
            got = sim.reduce(sp.FREE_ENERGY)
        with np.errstate(all="ignore"):
            ref = densities(q, h, c1, 1.0, 0.5, 0, sp).sum() * ((h * h) * h if len(shape) == 3 else h * h)
        assert got == ref or abs(got - ref) <= 1e-13 * abs(ref) or (np.isnan(got) and np.isnan(ref)), (dtype, got, ref)
