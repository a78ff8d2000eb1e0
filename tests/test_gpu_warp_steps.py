"""2D FP32 on warp rows: several steps per launch are bit for bit the single steps, and the generated
stencils the per-point kernels."""
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


# aligned and ragged rows of one strip, its edges (112 or 120 columns), and the sizes from which
# wide stencils take warp rows
@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(3, 4), (5, 1), (40, 120), (33, 121), (17, 242), (2051, 4100), (2049, 4098), (2050, 4097)])
def test_generated_rows(sp, model, order, shape):
    def go(cfg):
        kw = dict(seed=5, ic_amp=0.4)
        if model == 2:
            kw = dict(seed=5, ic_amp=0.05, gs_patches=2, gs_patch=1)
        with sp.Simulation(model, shape, dt=DT[model], stencil=sp.LAP_GENERATED, stencil_order=order, dtype=1, **kw) as s:
            s.launch_config = cfg
            s.step(3)
            return [s.read(f) for f in range(s.nfields)]

    for x, y in zip(go((1, 1)), go((1, 0))):
        assert np.isfinite(x).all() and np.array_equal(x, y)
