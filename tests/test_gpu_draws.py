"""The relabeling-draw kernels against the oracle's stream and each other (integers: equal,
no tolerance): words and steps that end inside a window (n around 32, 64, 256), one row on
a side, groups of columns that straddle a multiple of 2^32 draws (their words are
decided from whole Philox words), and enough slots that some words are too close to
call from the high halves (one slot in 2^21 for the lane kernels, n / 2^32 for the
warp kernel)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    c = ept.Context(0)
    c.set_option("autotune", 0)
    yield c
    c.close()


@pytest.mark.parametrize("nx,ny,b0,count", [
    (1, 31, 1, 70), (16, 17, 5, 33), (63, 1, 1, 40), (64, 192, 0, 65), (200, 57, 3, 300), (255, 258, 1, 129),
    (1000, 1001, 2**32 - 20, 40), (3000, 2000, 7, 3000)])
def test_warp_draws_equal_the_oracle(ctx, nx, ny, b0, count):
    got = ctx.perm_masks(11, nx, ny, b0, count)
    assert np.array_equal(got, oracle.pack_masks(oracle.perm_select(11, nx, ny, b0, count)))


@pytest.mark.parametrize("nx,ny,b0,count", [
    (1, 31, 1, 70), (16, 17, 5, 33), (63, 1, 1, 40), (64, 192, 1, 255), (57, 200, 3, 256), (255, 258, 1, 513),
    (500, 301, 2**32 - 20, 40), (3000, 2000, 7, 4000)])
def test_lane_draws_equal_the_warp_draws(ctx, nx, ny, b0, count):
    # the statistics of caller masks are the warp kernel's bits; the others must give the same
    rng = np.random.default_rng(3)
    X = rng.standard_normal((nx, 3), dtype=np.float32)
    Y = rng.standard_normal((ny, 3), dtype=np.float32)
    want = ctx.test_masks(X, Y, ctx.perm_masks(11, nx, ny, b0, count))
    for mode in (1, 2, 3):
        ctx.set_option("draw_mode", mode)
        try:
            got = ctx.test_range(X, Y, b_first=b0, count=count, seed=11)
        finally:
            ctx.set_option("draw_mode", 0)
        assert got.observed == want.observed and np.array_equal(got.stats, want.stats), mode
