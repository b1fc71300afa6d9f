"""Calls that use the context's scratch memory for something else between two runs of one
plan: the second run finds its tables and unit records again (the masks of ept_perm_masks
and the blocks of ept_build_blocks overwrite them) and returns the bits of the first."""
import numpy as np
import pytest

from paper_2406_06488_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    with ept.Context(0) as c:
        yield c


@pytest.mark.parametrize("graphs", [0, 1])
@pytest.mark.parametrize("between", ["perm_masks", "build_blocks", "perm_masks_small"])
def test_same_plan_after_another_use_of_the_scratch(ctx, between, graphs):
    ctx.set_option("graphs", graphs)
    X, Y = workloads.gaussian_pair(workloads.TwoSampleSpec(nx=300, ny=400, p=20, y_mean=0.1, data_seed=2))
    first = ctx.test(X, Y, B=700, seed=3)
    for _ in range(2):
        if between == "build_blocks":
            ctx.build_blocks(X[:250], Y[:260])
        else:
            ctx.perm_masks(5, 600, 500, 1, 20 if between.endswith("small") else 4000)
        again = ctx.test(X, Y, B=700, seed=3)
        assert again.observed == first.observed and again.n_ge == first.n_ge
        assert np.array_equal(again.stats, first.stats)
