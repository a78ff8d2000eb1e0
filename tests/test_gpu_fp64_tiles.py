"""3D FP64 kernels where the tile and the split of the planes change: grids that the
32 x 32 (64 x 32) tile covers exactly and badly (then 32 x 16 tiles are used), runs of
one plane, a run that crosses from one tile into the next, and grids smaller than a
tile.  Every family executes the oracle's operations in its order, so the tolerance is
zero."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


@pytest.mark.parametrize("st", [3, 4, 5])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 16, 33), (7, 32, 64), (5, 35, 71), (41, 47, 48), (700, 5, 6)])
def test_fp64_tiles_equal_oracle(sp, model, st, shape):
    dt, kw = 0.001, dict(seed=5, ic_amp=0.4)
    if model == 2:
        kw.update(ic_amp=0.01, gs_patches=2, gs_patch=1)
    with sp.Simulation(model, shape, dt=dt, stencil=st, **kw) as sim:
        f = [sim.read(i) for i in range(sim.nfields)]
        sim.step(3)
        got = [sim.read(i) for i in range(sim.nfields)]
    ref = O.step(model, st, *f, dt=dt, nsteps=3)
    for a, b in zip(got, ref if isinstance(ref, tuple) else (ref,)):
        assert np.array_equal(a, b)
