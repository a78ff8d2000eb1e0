"""The copy of a large served result: four threads share it, fewer where a thread cannot be started
(a limit on threads, an interpreter that is shutting down)."""
import threading

import numpy as np
import pytest


@pytest.mark.parametrize("most", [0, 1, 3, 100])
@pytest.mark.parametrize("n", [7, (2 << 20) + 3, 3 << 20])
def test_copy_without_threads(monkeypatch, n, most):
    import __graft_entry__

    __graft_entry__._load_builder().build()
    import paper_2511_10508_gb300 as sp

    started = []
    start = threading.Thread.start

    def limited(self):
        if len(started) >= most:
            raise RuntimeError("can't start new thread")
        started.append(self)
        start(self)

    monkeypatch.setattr(threading.Thread, "start", limited)
    src = np.random.default_rng(n).random(n)
    got = sp._copy(src)
    assert got is not src and np.array_equal(got, src)
    assert not any(t.is_alive() for t in started)
