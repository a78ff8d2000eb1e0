"""FP32 kernels on grids whose rows are not 16-byte aligned (nx odd, or 2 mod 4), and the row
and plane splits of small grids: rows shorter than a warp's 120 outputs, just above them,
and several strips; every model and stencil.  Families evaluate the same expressions in
the same order, so the default must equal the tile / staged family bit for bit, and fused
steps single ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


def run(sp, model, shape, st, dtype, cfg, steps=7):
    kw = dict(seed=9, ic_amp=0.3)
    if model == 2:
        kw = dict(seed=9, ic_amp=0.01, gs_patches=3, gs_patch=min(3, *shape))
    with sp.Simulation(model, shape, dt=0.001, stencil=st, dtype=dtype, **kw) as s:
        if cfg:
            s.launch_config = cfg
        s.step(steps)
        return [s.read(f) for f in range(s.nfields)]


@pytest.mark.parametrize("st", [0, 1, 2])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1), (3, 5), (40, 7), (9, 121), (70, 123), (33, 250), (5, 963), (64, 120), (300, 4)])
def test_2d_rows(sp, model, st, shape):
    a = run(sp, model, shape, st, 1, (1, 0))
    for cfg in ((1, 1), (2, 0), None):
        for x, y in zip(a, run(sp, model, shape, st, 1, cfg)):
            assert np.array_equal(x, y), cfg


@pytest.mark.parametrize("st", [3, 4, 5])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (9, 10, 121), (5, 17, 130), (40, 9, 7), (6, 33, 245), (7, 8, 120), (3, 17, 58), (2, 3, 2)])
def test_3d_rows(sp, model, st, shape):
    a = run(sp, model, shape, st, 1, None)
    for x, y in zip(a, run(sp, model, shape, st, 1, (1, 2))):  # staged planes (Model C: boxes)
        assert np.array_equal(x, y)


@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(64, 64), (257, 257), (256, 256), (80, 856), (411, 411), (31, 33)])
def test_2d_fp64_default_equals_single_steps(sp, model, shape):
    for x, y in zip(run(sp, model, shape, 0, 0, None), run(sp, model, shape, 0, 0, (1, 0))):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("dtype", [1, 2])
@pytest.mark.parametrize("st", [3, 4])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (9, 12, 120), (5, 13, 130), (40, 9, 7), (3, 25, 245), (7, 8, 124), (2, 3, 2)])
def test_model_h_rows(sp, st, shape, dtype):
    """Warp rows against the two per-point passes (tiles of 12 rows x 120 cells)."""
    def go(fam):
        kw = dict(flags=sp.FLAG_BF16_NO_BOUND) if dtype == 2 else {}
        with sp.Simulation(sp.MODEL_H, shape, dt=0.001, stencil=st, dtype=dtype, seed=4, ic_amp=0.5, **kw) as s:
            s.launch_config = (1, fam)
            s.step(5)
            return [s.read(f) for f in range(4)]
    for x, y in zip(go(0), go(1)):
        assert np.array_equal(x, y)


GEN_DT = {0: 0.02, 1: 0.001, 2: 0.2, 3: 0.01}


@pytest.mark.parametrize("order", [2, 4, 6, 8])
@pytest.mark.parametrize("model", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (9, 16, 56), (5, 17, 60), (40, 9, 7), (4, 33, 113), (3, 8, 57), (4, 9, 62), (2, 3, 2)])
def test_generated_3d_rows(sp, model, order, shape):
    """Row tiles (56 x 16) of the generated 3D stencils against the FP64 oracle started from
    the same rounded field: 3 steps of at most ~80 FP32 roundings (6e-8 each) of values of
    order 1 leave 2e-5; order 2 has the 7-point stencil's expressions and must equal it bit
    for bit."""
    import oracle as O

    kw = dict(seed=3, ic_amp=0.4)
    if model == 2:
        kw = dict(seed=3, ic_amp=0.05, gs_patches=2, gs_patch=1)
    with sp.Simulation(model, shape, dt=GEN_DT[model], stencil=sp.LAP_GENERATED, stencil_order=order, dtype=1, **kw) as s:
        ic = [s.read(f) for f in range(s.nfields)]
        s.step(3)
        got = [s.read(f) for f in range(s.nfields)]
    ref = O.step_gen(model, order, *ic, dt=GEN_DT[model], nsteps=3)
    for g, r in zip(got, ref if isinstance(ref, tuple) else (ref,)):
        assert np.abs(g - r).max() <= 2e-5
    if order == 2:
        with sp.Simulation(model, shape, dt=GEN_DT[model], stencil=sp.LAP_7, dtype=1, **kw) as s:
            s.step(3)
            for f, g in enumerate(got):
                assert np.array_equal(g, s.read(f))
