"""The tensor-core block build at the edges of its tiles, stages and epilogue, entry by
entry against the FP64 oracle: features around one stage of 32 (the last stage is zero
padding), rows around the 256-row panels, kernel values that are exactly 0 or mixed with
normal ones in one group of 32 columns, equal rows, close rows, and rows scaled so that
squared differences leave FP32's range.

Tolerances: the split Gram is good to 2^-20 of ||x||^2 + ||y||^2, which moves a distance d
by at most 2^-20 (||x||^2 + ||y||^2) / (2 d) and a kernel value by that times its
derivative; close rows are recomputed directly (every rounding below 2^-22 of the
entry, and no Gram error); 2^-21 of the entry covers the square root's and exp's roundings."""
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
    yield c
    c.close()


def _compare(ctx, X, Y, stat, sigma):
    got = ctx.build_blocks(X, Y, stat=stat, sigma=sigma).astype(np.float64)
    Z = np.concatenate([X, Y]).astype(np.float64)
    D = np.sqrt(((Z[:, None, :] - Z[None, :, :]) ** 2).sum(axis=2))
    n2 = (Z ** 2).sum(axis=1)
    sn = n2[:, None] + n2[None, :]
    close = D * D < 0.2 * sn    # well inside the recomputed set (d^2 < sn / 4)
    dd = np.where(close, 0.0, 2.0 ** -20 * sn / (2.0 * np.where(close, 1.0, D)))
    if stat == "ed":
        want, tol = D, dd
    elif stat == "mmd":
        want = np.exp(-D * D / (2.0 * sigma * sigma))
        tol = want * dd * D / sigma ** 2
    else:
        want = np.exp(-D / sigma)
        tol = want * dd / sigma
    tol = tol + 2.0 ** -21 * want * (1.0 + (0.0 if stat == "ed" else np.abs(np.log(np.maximum(want, 1e-38)))))
    err = np.abs(got - want)
    floor = 2.0 ** -125 if stat != "ed" else 0.0   # values below exp(-87) are written as 0
    assert (err <= tol + floor).all(), (float((err - tol).max()), np.unravel_index((err - tol).argmax(), err.shape))
    return got, want


@pytest.mark.parametrize("stat", ["ed", "mmd", "mmd_laplace"])
@pytest.mark.parametrize("nx,ny,p", [(1, 1, 1), (100, 156, 31), (128, 129, 32), (255, 2, 33), (200, 313, 64),
                                     (300, 212, 65), (40, 30, 200)])
def test_entries_at_tile_edges(ctx, nx, ny, p, stat):
    rng = np.random.default_rng(nx + p)
    X = rng.standard_normal((nx, p), dtype=np.float32)
    Y = rng.standard_normal((ny, p), dtype=np.float32) + np.float32(0.2)
    _compare(ctx, X, Y, stat, float(np.sqrt(p)))


@pytest.mark.parametrize("stat", ["mmd", "mmd_laplace"])
def test_kernel_values_of_zero(ctx, stat):
    rng = np.random.default_rng(5)
    X = rng.standard_normal((70, 4), dtype=np.float32)
    Y = rng.standard_normal((90, 4), dtype=np.float32)
    X[::7] += np.float32(60.0)   # far from the rest: those pairs' kernel values vanish, their neighbours' do not
    got, want = _compare(ctx, X, Y, stat, 0.6 if stat == "mmd" else 1.2)
    assert (got == 0.0).any() and (got > 0.0).any()
    assert (got[want < 1e-39] == 0.0).all()


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e18])
@pytest.mark.parametrize("stat", ["ed", "mmd"])
def test_equal_and_close_rows(ctx, scale, stat):
    rng = np.random.default_rng(6)
    X = (rng.standard_normal((80, 9)) * scale).astype(np.float32)
    Y = (rng.standard_normal((60, 9)) * scale).astype(np.float32)
    Y[:20] = X[:20]
    Y[20:40] = X[20:40] * np.float32(1.0 + 2.0 ** -18)
    got, want = _compare(ctx, X, Y, stat, 3.0 * scale)
    same = np.arange(20)
    assert (got[same, 80 + same] == (0.0 if stat == "ed" else 1.0)).all()


@pytest.mark.parametrize("stat", ["ed", "mmd"])
@pytest.mark.parametrize("nx,ny", [(300, 500), (800, 700), (1000, 1048), (1000, 1049), (1100, 1200)])
def test_tiles_shared_by_several_blocks(ctx, nx, ny, stat):
    """A quarter, half or all of a tile's columns to a thread block (up to 38, up to 76 and more tiles on 152
    SMs).  The row and column sums show in the statistic of the stored entries: the centred entries (at most
    16 times the largest) are packed to 2^-22, and no statistic's weights sum to more than 4; a K-block's
    missing sum would move it by more than 1e-3."""
    p = 5
    rng = np.random.default_rng(nx)
    X = rng.standard_normal((nx, p), dtype=np.float32)
    Y = rng.standard_normal((ny, p), dtype=np.float32) + np.float32(0.3)
    sigma = float(np.sqrt(p))
    got, _ = _compare(ctx, X, Y, stat, sigma)
    xx, yy, xy = got[:nx, :nx].sum() / nx ** 2, got[nx:, nx:].sum() / ny ** 2, got[:nx, nx:].sum() / (nx * ny)
    want = 2.0 * xy - xx - yy if stat == "ed" else xx + yy - 2.0 * xy
    r = ctx.test(X, Y, B=30, seed=1, stat=stat, sigma=sigma)
    assert abs(r.observed - want) <= 4.0 * 16.0 * 2.0 ** -22 * got.max()
