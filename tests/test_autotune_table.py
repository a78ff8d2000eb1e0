"""The autotuner's table: a choice measured on one grid is taken by another of its class
only where that grid has it.  Two steps per pass (3D FP32) and tensor-map loads need rows
that are multiples of 4 values; grids with other rows in the same class of sizes have
neither."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


def _args(sp, model, shape, dtype):
    prm = sp.params(model, len(shape), dtype=dtype)
    xyz = (ctypes.c_int64 * 3)(*(list(shape[::-1]) + [1] * (3 - len(shape))))
    return model, len(shape), xyz, ctypes.byref(prm)


def record(sp, model, shape, dtype, choice):
    return sp.N.lib().sp_tune_record(*_args(sp, model, shape, dtype), *choice)


def lookup(sp, model, shape, dtype):
    spl, var = ctypes.c_int(-1), ctypes.c_int(-1)
    rc = sp.N.lib().sp_tune_lookup(*_args(sp, model, shape, dtype), ctypes.byref(spl), ctypes.byref(var))
    assert rc in (sp.N.SP_OK, sp.N.SP_ENOTFOUND)
    return (spl.value, var.value) if rc == sp.N.SP_OK else None


@pytest.mark.parametrize("choice", [(2, 0), (2, 1)])
@pytest.mark.parametrize("model", [0, 2, 3])
def test_two_steps_per_pass_stay_with_aligned_rows(sp, model, choice):
    """(44, 44, 44) and the others have between 2^16 and 2^17 points."""
    assert record(sp, model, (44, 44, 44), 1, choice) == sp.N.SP_OK
    for nx in (41, 42, 43, 45, 46, 47):
        assert lookup(sp, model, (44, 44, nx), 1) != choice
        assert record(sp, model, (44, 44, nx), 1, choice) == sp.N.SP_EINVAL
    assert lookup(sp, model, (40, 48, 44), 1) == choice


def test_small_grid_choice_stays_with_small_grids(sp):
    """2D FP64 fuses four steps up to 1024^2 points; 1024 x 1032 is of the same power of two."""
    assert record(sp, 0, (1024, 1024), 0, (4, 0)) == sp.N.SP_OK
    assert lookup(sp, 0, (1024, 1024), 0) == (4, 0)
    assert lookup(sp, 0, (1032, 1024), 0) is None


@pytest.mark.gpu
@pytest.mark.parametrize("model", [0, 2, 3])
def test_unaligned_grid_after_an_aligned_winner(sp, model):
    """As an autotuned program meets it: an aligned grid's class holds two steps per pass, then
    grids of the same size with other rows autotune; every result equals single steps."""
    assert record(sp, model, (44, 44, 44), 1, (2, 0)) == sp.N.SP_OK
    kw = dict(dt=0.02, dtype=sp.F32, seed=3)
    if model == 2:
        kw.update(gs_patches=2, gs_patch=6)
    for nx in (44, 42, 43):
        with sp.Simulation(model, (44, 44, nx), steps_per_launch=1, **kw) as a, \
                sp.Simulation(model, (44, 44, nx), flags=sp.FLAG_AUTOTUNE, **kw) as b:
            a.step(80)
            b.step(80)
            assert b.launch_config[0] == (2 if nx == 44 else 1)
            for f in range(a.nfields):
                assert np.array_equal(a.read(f), b.read(f))
