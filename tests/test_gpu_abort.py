"""A block build whose wait expires gives up as a whole.  The hook makes one of its epilogue
warps wait out the limit on a flag that nothing sets while the tiles' accumulators still
complete, so that the warps that share its half of a tile's columns go on for a tile or two
without it: with one tile or part of a tile per thread block, with several, with tests that
take their sums elsewhere (a median bandwidth) in between, and in windows.  The call returns
EPT_ETIMEOUT within a few limits, and the next run of the context is right.  The same for the
contraction kernels, whose stalled issuer leaves every stage's copies and relabeling tiles done or
under way."""
import time

import numpy as np
import pytest

from paper_2406_06488_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    c = ept.Context(0)
    c.set_option("autotune", 0)
    c.set_option("wait_limit_ms", 50)
    yield c
    c.close()


def _pair(nx, ny, p, seed):
    return workloads.gaussian_pair(workloads.TwoSampleSpec(nx=nx, ny=ny, p=p, y_mean=0.2, data_seed=seed))


def _expires(ctx, call, hook=2):
    from paper_2406_06488_gb300 import ept
    ctx.set_option("fault_inject_stall", hook)
    t0 = time.perf_counter()
    with pytest.raises(ept.EptError) as e:
        call()
    assert e.value.status == 5
    assert time.perf_counter() - t0 < 2.0


@pytest.mark.parametrize("nx,ny,p", [(70, 60, 3), (300, 400, 33), (900, 1100, 8), (2600, 2400, 20), (6000, 6100, 40)])
def test_build_gives_up_as_a_whole(ctx, nx, ny, p):
    X, Y = _pair(nx, ny, p, seed=nx)
    want = ctx.test(X, Y, B=60, seed=2)
    _expires(ctx, lambda: ctx.test(X, Y, B=60, seed=2))
    got = ctx.test(X, Y, B=60, seed=2)
    assert got.observed == want.observed and np.array_equal(got.stats, want.stats)


def test_build_gives_up_in_a_batch(ctx):
    tests = []
    for k in range(60):
        X, Y = _pair(200 + 11 * k, 300, 6, seed=k)
        tests.append(dict(X=X, Y=Y, B=20, seed=k, stat="mmd", sigma="median" if k % 3 == 1 else 2.0))
    want = ctx.test_batch(tests)
    _expires(ctx, lambda: ctx.test_batch(tests))
    for a, b in zip(want, ctx.test_batch(tests)):
        assert a.observed == b.observed and a.n_ge == b.n_ge


def test_build_gives_up_in_windows(ctx):
    X, Y = _pair(2000, 2100, 9, seed=5)
    try:
        ctx.set_option("stream_blocks", 300)
        want = ctx.test(X, Y, B=40, seed=3)
        assert want.n_windows > 2
        _expires(ctx, lambda: ctx.test(X, Y, B=40, seed=3))
        got = ctx.test(X, Y, B=40, seed=3)
        assert got.observed == want.observed and np.array_equal(got.stats, want.stats)
    finally:
        ctx.set_option("stream_blocks", 0)


@pytest.mark.parametrize("kernel", [1, 2, 3])
@pytest.mark.parametrize("nx,ny,B", [(60, 70, 30), (2600, 2400, 1500)])   # one unit of few K-blocks, and many units
def test_contraction_gives_up(ctx, kernel, nx, ny, B):
    X, Y = _pair(nx, ny, 12, seed=nx)
    try:
        ctx.set_option("contraction", kernel)
        want = ctx.test(X, Y, B=B, seed=4)
        for _ in range(3):
            _expires(ctx, lambda: ctx.test(X, Y, B=B, seed=4), hook=1)
            got = ctx.test(X, Y, B=B, seed=4)
            assert got.observed == want.observed and np.array_equal(got.stats, want.stats)
    finally:
        ctx.set_option("contraction", 0)


def test_build_blocks_reports_an_expired_wait(ctx):
    X, Y = _pair(700, 900, 5, seed=9)
    want = ctx.build_blocks(X, Y)
    _expires(ctx, lambda: ctx.build_blocks(X, Y))
    assert np.array_equal(ctx.build_blocks(X, Y), want)
