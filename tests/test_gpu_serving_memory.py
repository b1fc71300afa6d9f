"""An idle server gives the memory of its requests' samples back: after a burst of 40 MB requests and a
pause past the two seconds for which it is kept, the process holds less by nearly all of it."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _resident():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) * 1024 for line in f if line.startswith("VmRSS"))


def test_idle_server_gives_sample_memory_back():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    rng = np.random.default_rng(0)
    X, Y = rng.standard_normal((2000, 2500), dtype=np.float32), rng.standard_normal((2000, 2500), dtype=np.float32)
    with ept.Context(0) as ctx:
        for _ in range(2):
            for t in [ctx.submit(X, Y, B=20, seed=k) for k in range(5)]:
                ctx.wait(t)
        held = _resident()
        time.sleep(4.0)
        assert held - _resident() >= 150 << 20   # five requests of 40 MB, the rest left to the allocator
        one = ctx.wait(ctx.submit(X, Y, B=20, seed=3))
        assert np.abs(one.stats - ctx.test(X, Y, B=20, seed=3).stats).max() <= 1e-6 * abs(one.observed)
