"""Requests whose samples are copied by the worker threads, or into memory that an earlier
request has used: sizes around the line for the workers (2^20 bytes) and for kept memory
(2^17), several threads submitting at once, new data every time.  Each answer is that of the
same test run alone: whole numbers equal, statistics to 1e-6 of their spread plus the observed
value (a batch may sum the same FP32 entries over other units)."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(3, 5, 2), (180, 76, 128), (180, 76, 127), (1000, 48, 250), (1000, 49, 250), (1200, 1100, 301), (1300, 1201, 300)]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    c = ept.Context(0)
    c.set_option("autotune", 0)
    yield c
    c.close()


def _data(k, seed):
    nx, ny, p = SHAPES[k]
    r = np.random.default_rng(100 * seed + k)
    return r.standard_normal((nx, p), dtype=np.float32), r.standard_normal((ny, p), dtype=np.float32) + np.float32(0.1)


@pytest.mark.parametrize("threads", [1, 4])
def test_reused_memory_holds_the_new_samples(ctx, threads):
    got, errors = {}, []

    def client(w):
        try:
            for rep in range(3):
                seeds = [10 * w + rep] * len(SHAPES)
                tickets = []
                for k, s in enumerate(seeds):
                    X, Y = _data(k, s)
                    tickets.append(ctx.submit(X, Y, B=60, seed=s))
                    X.fill(np.nan)    # the request has its own copy
                    Y.fill(np.nan)
                order = list(range(len(SHAPES)))
                for k in order[::-1] if rep % 2 else order:
                    got[k, seeds[k]] = ctx.wait(tickets[k])
        except Exception as e:   # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=client, args=(w,)) for w in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
    for (k, s), g in got.items():
        one = ctx.test(*_data(k, s), B=60, seed=s)
        assert g.n_ge == one.n_ge and g.p_value == one.p_value
        tol = 1e-6 * (np.std(one.stats) + abs(one.observed))
        assert abs(g.observed - one.observed) <= tol
        assert np.abs(g.stats - one.stats).max() <= tol
