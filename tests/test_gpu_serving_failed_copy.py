"""A request whose result cannot be copied to the host: it fails, gives no fields (host memory that
nothing wrote), and the server goes on."""
import ctypes
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


@pytest.mark.parametrize("dtype", [0, 1])
def test_failed_copy_gives_no_fields(sp, dtype):
    kw = dict(dt=0.05, nsteps=30, seed=9, dtype=dtype, return_fields=True)
    with sp.Server(1 << 30) as srv:
        bad = srv.submit(0, (64, 96), fault=2, **kw)
        good = srv.submit(0, (64, 96), **kw)
        fields = srv.wait(good).fields
        end = time.time() + 60
        res = sp.N.sp_result()
        while sp.N.lib().sp_poll(srv._h, bad, ctypes.byref(res)) == sp.N.SP_PENDING and time.time() < end:
            time.sleep(0.01)
        assert res.status == sp.N.SP_ECUDA and not res.fields and res.n_values == 0 and res.mass == 0.0
        with pytest.raises(sp.SpError):
            srv.wait(bad)
        again = srv.wait(srv.submit(0, (64, 96), **kw))
    assert np.isfinite(fields).all() and np.array_equal(again.fields, fields)
