"""Row sums and centring in one launch (tests of up to 1,024 padded rows) against the three kernels of larger
ones: each small test alone, and in a batch with one test of 1,025 rows, which takes the whole batch there.

Tolerance: both sum the same FP64 terms in another order (2^-45 of them), which may move a u_i by one
FP32 rounding; the statistic is the same for any u but for the packing of the centred entries, 2^-22 of at
most 16 times the largest entry, and no statistic's weights sum to more than 4."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("prec", ["split_bf16", "plain_fp32"])
def test_one_launch_equals_three(ctx, prec):
    rng = np.random.default_rng(4)
    tests = []
    for k, (nx, ny) in enumerate([(1, 1), (30, 2), (100, 156), (129, 128), (255, 257), (256, 257), (400, 368), (500, 269),
                                  (511, 513), (1000, 24), (512, 513)]):
        X = rng.standard_normal((nx, 7), dtype=np.float32)
        Y = rng.standard_normal((ny, 7), dtype=np.float32) + np.float32(0.2)
        tests.append(dict(X=X, Y=Y, B=70, seed=k, stat="mmd" if k % 3 == 1 else "ed", sigma=2.5))
    small, big = tests[:-1], tests
    assert all(len(t["X"]) + len(t["Y"]) <= 1024 for t in small) and len(big[-1]["X"]) + len(big[-1]["Y"]) == 1025
    one = ctx.test_batch(small, prec=prec)
    three = ctx.test_batch(big, prec=prec)
    for t, a, b in zip(small, one, three):
        Z = np.concatenate([t["X"], t["Y"]]).astype(np.float64)
        top = 1.0 if t["stat"] == "mmd" else np.sqrt(((Z[:, None] - Z[None]) ** 2).sum(axis=2)).max()
        tol = 4.0 * 16.0 * 2.0 ** -22 * top
        assert abs(a.observed - b.observed) <= tol
        assert np.abs(np.asarray(a.stats) - np.asarray(b.stats)).max() <= tol
        alone = ctx.test(t["X"], t["Y"], B=70, seed=t["seed"], stat=t["stat"], sigma=2.5, prec=prec)
        assert abs(alone.observed - a.observed) <= tol
