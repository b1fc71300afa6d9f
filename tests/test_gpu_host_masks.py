"""Caller relabelings in host memory: the kernel that reads them waits for their copy
(it runs on its own stream, beside the copies of X and Y), so a call sees its own
relabelings and not what an earlier call left in the scratch memory."""
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
    yield c
    c.close()


@pytest.mark.parametrize("path", ["replayed", "direct", "streaming", "pooled_fp32"])
def test_host_masks_are_the_calls_own(ctx, path):
    nx, ny, p, B = 1900, 2300, 700, 1500   # 12 MB of rows ahead of the relabelings in the copy queue
    X, Y = workloads.gaussian_pair(workloads.TwoSampleSpec(nx=nx, ny=ny, p=p, y_mean=0.02, data_seed=4))
    prec = path if path == "pooled_fp32" else "split_bf16"
    ctx.set_option("graphs", 0 if path == "direct" else 1)
    ctx.set_option("stream_blocks", 200 if path == "streaming" else 0)
    try:
        for seed in (1, 2, 3):
            masks = ctx.perm_masks(seed, nx, ny, 1, B)
            got = ctx.test_masks(X, Y, masks, prec=prec)
            want = ctx.test(X, Y, B=B, seed=seed, prec=prec)
            assert got.observed == want.observed and got.n_ge == want.n_ge
            assert np.array_equal(got.stats, want.stats)   # the same kernels on the same relabelings
    finally:
        ctx.set_option("graphs", 1)
        ctx.set_option("stream_blocks", 0)
