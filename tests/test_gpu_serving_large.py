"""Served grids of a million points and more, which are stepped by the single-grid kernels
beside the batched launches: every result equals the same grid run alone, bit for bit,
for step counts that end inside a quantum, odd counts with two steps per launch, and a
quantum of odd length (the levels then change sides from quantum to quantum)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


# (model, shape, dtype, stencil, dt, steps); the smallest is just above 2^20 points, two are small
MIX = [(2, (1025, 1024), 1, 0, 0.5, 23), (0, (1031, 1033), 0, 1, 0.05, 8), (1, (1100, 1000), 1, 2, 0.002, 17),
       (1, (101, 103, 102), 0, 3, 0.002, 9), (1, (128, 96, 100), 1, 5, 0.001, 15), (2, (110, 100, 100), 0, 4, 0.2, 7),
       (3, (104, 104, 104), 1, 3, 0.02, 11), (1, (102, 102, 102), 0, 4, 0.002, 5), (0, (60, 70), 0, 0, 0.05, 21),
       (1, (20, 30, 40), 1, 3, 0.002, 30)]


@pytest.mark.parametrize("quantum", [6, 5])
def test_large_served_grids_equal_alone(sp, quantum):
    def kw(i, m):
        return dict(seed=40 + i, ic_amp=0.01 if m == 2 else 0.3, **(dict(gs_patches=3, gs_patch=8) if m == 2 else {}))

    with sp.Server(8 << 30, max_slots=16, quantum_steps=quantum) as srv:
        for _ in range(2):  # again on the same server: graphs, tables and streams are reused
            t = [srv.submit(m, sh, dt=dt, nsteps=n, stencil=st, dtype=ty, return_fields=True, **kw(i, m))
                 for i, (m, sh, ty, st, dt, n) in enumerate(MIX)]
            for i, ((m, sh, ty, st, dt, n), res) in enumerate(zip(MIX, [srv.wait(x, timeout=300) for x in t])):
                assert res.steps_done == n
                with sp.Simulation(m, sh, dt=dt, stencil=st, dtype=ty, **kw(i, m)) as s:
                    s.step(n)
                    for f in range(s.nfields):
                        assert np.array_equal(res.fields[f], s.read(f)), (i, f)
