"""The median heuristic's selection is exact: the bandwidth is the lower median of the FP32
distances as built (the same kernel writes them for ept_build_blocks), bit for bit.
Cases: sizes whose sample is too small to bracket the median (the selection starts from all
values), panel and block edges, ties, distances over many binades, two clusters with
the median at the edge of the gap, and several tests in one batch."""
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


def _rows(kind, n, p, rng):
    Z = rng.standard_normal((n, p)).astype(np.float32)
    if kind == "ties":
        Z = rng.integers(0, 3, (n, p)).astype(np.float32)
    elif kind == "binades":
        Z *= np.exp2(rng.uniform(-12, 12, (n, 1))).astype(np.float32)
    elif kind == "clusters":
        Z[: n // 2] += np.float32(100.0)
    return Z


def _want(ctx, X, Y):
    D = ctx.build_blocks(X, Y, stat="ed")
    d = np.sort(D[np.triu_indices(D.shape[0], 1)])
    return d[(d.size - 1) // 2]


@pytest.mark.parametrize("kind", ["normal", "ties", "binades", "clusters"])
@pytest.mark.parametrize("nx,ny,p", [(1, 1, 3), (2, 3, 2), (20, 21, 5), (100, 156, 8), (200, 57, 33), (700, 813, 6),
                                     (1300, 1260, 40)])
def test_bandwidth_is_the_lower_median(ctx, kind, nx, ny, p):
    Z = _rows(kind, nx + ny, p, np.random.default_rng(nx * 31 + ny))
    X, Y = Z[:nx], Z[nx:]
    want = _want(ctx, X, Y)
    if not want > 0:
        pytest.skip("more than half of the pairs coincide")
    got = ctx.test(X, Y, B=20, seed=1, stat="mmd", sigma="median")
    assert got.sigma == float(want)


def test_bandwidths_of_a_batch(ctx):
    rng = np.random.default_rng(9)
    tests = []
    for k, (nx, ny, p) in enumerate([(30, 40, 4), (600, 500, 20), (3, 2, 2), (256, 256, 7), (900, 1000, 3)]):
        Z = _rows(["normal", "binades", "normal", "ties", "clusters"][k], nx + ny, p, rng)
        tests.append(dict(X=Z[:nx], Y=Z[nx:], B=30, seed=k, stat="mmd" if k % 2 else "mmd_laplace", sigma="median"))
    tests.insert(2, dict(X=tests[0]["X"], Y=tests[0]["Y"], B=30, seed=7, stat="ed"))   # without a bandwidth
    for t, r in zip(tests, ctx.test_batch(tests)):
        if t["stat"] != "ed":
            assert r.sigma == float(_want(ctx, t["X"], t["Y"]))
