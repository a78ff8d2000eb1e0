"""The free-energy reduction where its chunks end: rows shorter and longer than a
16-byte chunk, sides that are no multiple of it, single rows and planes, and values
whose widening to FP64 takes another path (denormals, zeros of both signs, infinity).

Tolerance: at most 16 roundings touch a point's terms (u = 2^-53 each, relative to
their magnitudes): the differences and squares, the products, the sums of 8 points and
the compensated sum; the reference is computed in extended precision."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


def terms(fields, h, model, sp):
    """Point terms of the discrete energy (c1 = c2 = 1, c3 = 0.5) in extended precision."""
    q = [f.astype(np.longdouble) for f in fields]
    p = q[0]
    out = [-p * p / 2, p ** 4 / 4]
    for ax in range(p.ndim):
        d = np.roll(p, -1, ax) - p
        out.append(d * d / (2 * np.longdouble(h) ** 2))
    if model == sp.MODEL_C:
        out += [q[1] * q[1] / 2, -p * p * q[1] / 2]
    if model == sp.MODEL_H:
        out += [j * j / 2 for j in q[1:]]
    return out


@pytest.mark.parametrize("dtype", [0, 1, 2])
@pytest.mark.parametrize("model,shape", [(0, (1, 1)), (1, (1, 5)), (1, (3, 4)), (0, (5, 33)), (1, (130, 257)),
                                         (0, (1, 1, 3)), (1, (2, 3, 5)), (1, (4, 6, 8)), (0, (9, 17, 70)), (3, (7, 13)),
                                         (3, (3, 5, 9)), (4, (6, 10)), (4, (5, 4, 11))])
def test_energy_at_chunk_edges(sp, model, shape, dtype):
    h = 0.75
    rng = np.random.default_rng(11)
    with sp.Simulation(model, shape, h=h, dt=1e-4, dtype=dtype, flags=sp.FLAG_BF16_NO_BOUND if dtype == 2 else 0) as sim:
        for f in range(sim.nfields):
            v = rng.uniform(-1.5, 1.5, shape)
            v.ravel()[::5] = 0.0
            v.ravel()[1::7] = -0.0
            v.ravel()[2::6] = 3e-41  # denormal in FP32
            sim.write(f, v)
        t = terms([sim.read(f) for f in range(sim.nfields)], h, model, sp)
        got = sim.reduce(sp.FREE_ENERGY)
        vol = h ** len(shape)
        exact = float(sum(x.sum() for x in t) * vol)
        bound = 16 * U * float(sum(np.abs(x).sum() for x in t)) * vol
        assert abs(got - exact) <= bound, (got, exact, bound)
        v = sim.read(0)
        v.ravel()[v.size // 2] = np.inf
        sim.write(0, v)
        assert np.isnan(sim.reduce(sp.FREE_ENERGY))
