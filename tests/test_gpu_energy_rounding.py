"""The free energy's sum adds nothing to the roundings of the point densities: over many
fields its error has no mean.

u = 2^-53.  The result is rounded once (h = 1) or twice (the cell volume of h = 3/4 is exact),
each time by at most u of it and evenly, so the mean over 64 fields has a deviation below
sqrt(2) 0.58 u / 8 = 0.1 u; the squares of FP32 differences, whose last bits are not even, leave
up to 0.1 u (a host model of the point densities).  Bound 0.4 u.  Sums of 8 points in plain
FP64 leave 0.95 u (FP32, h = 1), a rounded 1/(2 h^2) 0.55 u (FP64, h = 3/4) in that model."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


@pytest.mark.parametrize("dtype,h", [(1, 1.0), (0, 1.0), (1, 0.75), (0, 0.75)])
def test_energy_error_has_no_mean(sp, dtype, h):
    off = []
    with sp.Simulation(0, (16, 16, 16), h=h, dt=1e-4, dtype=dtype) as sim:
        for seed in range(64):
            sim.write(0, np.random.default_rng(seed).uniform(-0.5, 0.5, (16, 16, 16)))
            p = sim.read(0).astype(np.longdouble)
            e = p ** 4 / 4 - p * p / 2
            for ax in range(3):
                d = np.roll(p, -1, ax) - p
                e = e + d * d / (2 * np.longdouble(h) ** 2)
            exact = e.sum() * np.longdouble(h) ** 3
            off.append(float((np.longdouble(sim.reduce(sp.FREE_ENERGY)) - exact) / exact) * 2.0 ** 53)
    assert abs(np.mean(off)) <= 0.4, off


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("shape", [(700, 700), (701, 703)])
@pytest.mark.parametrize("rising", [True, False])
def test_energy_of_fields_over_many_binary_orders(sp, dtype, shape, rising):
    """Magnitudes from 2^-40 to 2^30 (a thread's points rise or fall through them), zeros between.
    At most 16 roundings per term, as in test_gpu_energy.py."""
    n = shape[0] * shape[1]
    v = np.random.default_rng(5).uniform(-1, 1, n) * 2.0 ** np.linspace(-40, 30, n)
    v[::9] = 0.0
    v = (v if rising else v[::-1]).reshape(shape)
    with sp.Simulation(0, shape, dt=1e-4, dtype=dtype) as sim:
        sim.write(0, v)
        p = sim.read(0).astype(np.longdouble)
        got = sim.reduce(sp.FREE_ENERGY)
    terms = [-p * p / 2, p ** 4 / 4] + [(np.roll(p, -1, ax) - p) ** 2 / 2 for ax in range(2)]
    exact, size = float(sum(t.sum() for t in terms)), float(sum(np.abs(t).sum() for t in terms))
    assert abs(got - exact) <= 16 * 2.0 ** -53 * size
