"""The median bandwidth with more than 2^32 pairs in one bin of the selection: 100,000 rows of 40
categories (one-hot), whose 4.9 10^9 pairs of different categories are all at the distance sqrt(2) (exact
in the Gram expansion but for the square root, good to 2^-22)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_more_equal_distances_than_32_bits_count():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_06488_gb300 import ept
    import torch
    n = 100_000
    assert n * (n - 1) // 2 - 40 * (n // 40) ** 2 // 2 > 2 ** 32
    Z = torch.eye(40, device="cuda").repeat(n // 40, 1)
    with ept.Context(0) as ctx:
        ctx.set_option("autotune", 0)
        r = ctx.test(Z[: n // 2].contiguous(), Z[n // 2:].contiguous(), B=20, seed=1, stat="mmd", sigma="median")
    assert abs(r.sigma - np.sqrt(2.0)) <= 2.0 ** -22 * np.sqrt(2.0)
