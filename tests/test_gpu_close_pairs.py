"""Close pairs of rows (d^2 below a quarter of ||x||^2 + ||y||^2) hold what an FP64 sum of squared differences
gives, rounded once: few, ordinary, many and very many features, few enough rows that FP64 arithmetic on the
host decides every entry.  An entry may differ from the host's only where the FP64 value, within the two sums'
own 2^-53 p, lies at the middle between two FP32 numbers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    c = ept.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("stat", ["ed", "mmd", "mmd_laplace"])
@pytest.mark.parametrize("n,p", [(300, 1), (1500, 7), (1500, 10), (800, 130), (500, 1500), (600, 8000)])
def test_close_pairs_are_rounded_once(ctx, n, p, stat):
    rng = np.random.default_rng(p)
    # far from the origin: the features share a large part, so that every pair is close
    Z = (20.0 * rng.standard_normal(p) + 30.0 + rng.standard_normal((n, p))).astype(np.float32)
    sigma = 2.0 ** round(np.log2(np.sqrt(p) + 1.0))   # 1 / sigma and 1 / (2 sigma^2) are FP32 numbers
    got = ctx.build_blocks(Z[: n // 2], Z[n // 2:], stat=stat, sigma=sigma)
    Z64 = Z.astype(np.float64)
    for i in range(n - 1):
        S = np.zeros(n - 1 - i)
        for k in range(0, p, 1000):
            S += ((Z64[i + 1:, k:k + 1000] - Z64[i, k:k + 1000]) ** 2).sum(axis=1)
        v = {"ed": np.sqrt, "mmd": lambda s: np.exp(-s / (2.0 * sigma ** 2)),
             "mmd_laplace": lambda s: np.exp(-np.sqrt(s) / sigma)}[stat](S)
        # sums of n terms: p 2^-53 each; a kernel value's exponent is at most 90 here
        rel = (2.0 * p + 16.0) * 2.0 ** -53 * (0.5 if stat == "ed" else 90.0)
        lo, hi = (v * (1.0 - rel)).astype(np.float32), (v * (1.0 + rel)).astype(np.float32)
        g = got[i, i + 1:]
        assert ((g == lo) | (g == hi)).all(), (i, g[(g != lo) & (g != hi)], lo[(g != lo) & (g != hi)])
