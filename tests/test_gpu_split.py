"""The FP16 split and the row norms with eight lanes a row (many rows: a batch) against a warp a row
(the same test alone): features around one step of 4 and around a lane group's 32, rows that
start off a 16-byte boundary, norms near and past FP32's limit, and rows that are not finite.

Tolerance, in units of s = sqrt(largest squared norm): a norm is the same sum, good to 2^-40 and
rounded once, so it moves by 2^-23 of itself at most; pairs with d^2 < (N_i + N_j) / 4 are recomputed
without it, so an entry moves by at most 2^-23 sqrt(2) s, and 2^-23 s more in its own rounding.  The centred
entries (at most 16 s) are packed to 2^-22.  No statistic's weights sum to more than 4."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROWS_A_SIDE = 100    # 200 rows, padded to 256


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    c = ept.Context(0)
    c.set_option("autotune", 0)
    yield c
    c.close()


def _sample(rng, p, scale, off):
    import torch
    x = torch.from_numpy((rng.standard_normal(ROWS_A_SIDE * p) * scale).astype(np.float32)).cuda()
    buf = torch.empty(ROWS_A_SIDE * p + 4, dtype=torch.float32, device="cuda")
    buf[off:off + x.numel()] = x
    return buf[off:off + x.numel()].view(ROWS_A_SIDE, p)


@pytest.mark.parametrize("scale", [1.0, 1e-30, 0.7e18, 4e18])
@pytest.mark.parametrize("widths", [(1, 2, 3, 4, 5, 31, 32, 33, 64, 97, 100, 127, 128), (20, 129, 131, 256, 500, 512)])
def test_batch_equals_single(ctx, widths, scale):
    rng = np.random.default_rng(int(widths[-1]))
    count = 32 if widths[-1] <= 128 else 136    # 256 rows each: past the line of either rule
    tests = []
    for k in range(count):
        p = widths[k % len(widths)]
        tests.append(dict(X=_sample(rng, p, scale, k % 4), Y=_sample(rng, p, scale * 1.5, k // 2 % 4), B=40, seed=k))
    got = ctx.prepare_batch(tests).run()
    for t, g in list(zip(tests, got))[:2 * len(widths)]:
        one = ctx.test(t["X"], t["Y"], B=40, seed=t["seed"])
        a, b = np.asarray(g.stats.cpu()), np.asarray(one.stats.cpu())
        a, b = np.append(a, g.observed), np.append(b, one.observed)
        np.testing.assert_array_equal(np.isfinite(a), np.isfinite(b))
        Z = np.concatenate([t["X"].cpu().numpy(), t["Y"].cpu().numpy()]).astype(np.float64)
        N = (Z ** 2).sum(axis=1).max()
        tol = 4.0 * (2.0 ** -23 * (2.0 ** 0.5 + 1.0) + 2.0 ** -22 * 16.0) * np.sqrt(N)
        ok = np.isfinite(a)
        assert (np.abs(a - b)[ok] <= tol).all(), (t["X"].shape, np.abs(a - b)[ok].max(), tol)


def test_rows_that_are_not_finite_are_refused(ctx):
    rng = np.random.default_rng(3)
    tests = [dict(X=_sample(rng, 33, 1.0, 1), Y=_sample(rng, 33, 1.0, 0), B=20, seed=k) for k in range(32)]
    tests[17]["Y"][60, 32] = float("nan")
    tests[21]["X"][3, 0] = float("inf")
    with pytest.raises(Exception) as e:
        ctx.prepare_batch(tests).run()
    alone = None
    try:
        ctx.test(tests[17]["X"], tests[17]["Y"], B=20, seed=0)
    except Exception as x:
        alone = x
    assert type(alone) is type(e.value)
