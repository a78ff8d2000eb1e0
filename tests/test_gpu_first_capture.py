"""Graph-sized calls after other calls: single steps first (the kernel of several steps per launch
has then not run), and a launch configuration changed between calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sp():
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    return sp


@pytest.mark.parametrize("model,shape,dtype", [(0, (61, 90), 1), (3, (100, 64), 1), (0, (96, 96), 0), (1, (24, 20, 40), 1)])
def test_graph_sized_calls_after_single_steps(sp, model, shape, dtype):
    kw = dict(dt=0.005, dtype=dtype, seed=9)
    with sp.Simulation(model, shape, steps_per_launch=1, **kw) as a, sp.Simulation(model, shape, **kw) as b:
        for _ in range(170):
            a.step(1)
        for _ in range(5):
            b.step(1)
        b.step(65)
        first = b.launch_config
        b.launch_config = (1, 1) if len(shape) == 2 else (1, 2)
        b.step(50)
        b.launch_config = first if first[0] in (1, 2, 4) else (1, 0)
        b.step(50)
        for f in range(a.nfields):
            assert np.array_equal(a.read(f), b.read(f))
