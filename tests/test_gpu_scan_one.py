"""The exclusive scan on both sides of the size up to which one block does it, against a
cumulative sum, bit for bit, and in place."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 1023, 1024, 1025, 2047, 15 * 1024 + 1, 16383, 16384, 16385, 20_000])
def test_scan_sizes_of_one_block(n):
    from paper_2411_06224_gb300 import binding as B

    ctx = B.gs_create(0)
    x = np.random.default_rng(n).integers(-1000, 1000, n).astype(np.int32)
    want = np.concatenate([[0], np.cumsum(x, dtype=np.int64)[:-1]]).astype(np.int32)
    xd = torch.as_tensor(x, device="cuda")
    assert np.array_equal(B.gs_prim_exclusive_scan(ctx, xd).cpu().numpy(), want)
    B.gs_prim_exclusive_scan(ctx, xd, out=xd)
    assert np.array_equal(xd.cpu().numpy(), want)
    B.gs_destroy(ctx)
