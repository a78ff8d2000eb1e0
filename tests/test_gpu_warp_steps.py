"""2D FP32, several steps per launch on warp rows: bit for bit the single steps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DT = {0: 0.02, 1: 0.001, 2: 0.2, 3: 0.01}


@pytest.fixture(scope="module")
def sp():
    import paper_2511_10508_gb300 as m

    return m


# strips of 120 columns, two per CTA from 32 strips on; rows aligned to 16, 8 and 4 bytes
@pytest.mark.parametrize("st", [0, 1, 2])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1), (2, 4), (3, 2), (5, 120), (33, 124), (40, 241), (7, 3964), (19, 3963), (17, 3850)])
def test_steps_per_launch(sp, model, st, shape):
    def go(cfg):
        kw = dict(seed=5, ic_amp=0.4)
        if model == 2:
            kw = dict(seed=5, ic_amp=0.05, gs_patches=2, gs_patch=1)
        with sp.Simulation(model, shape, dt=DT[model], stencil=st, dtype=1, **kw) as s:
            if cfg:
                s.launch_config = cfg
            s.step(1)
            s.step(11)  # 4 + 4 + 2 + 1
            return [s.read(f) for f in range(s.nfields)]

    a = go((1, 0))
    assert all(np.isfinite(x).all() for x in a)
    for cfg in ((2, 0), (4, 0), None):
        for x, y in zip(a, go(cfg)):
            assert np.array_equal(x, y)
