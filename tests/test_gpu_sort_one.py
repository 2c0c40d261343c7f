"""Sorts of up to 8,192 pairs run in one block: sizes at its edges and numbers of digits
(odd and even, a last digit of one bit), against numpy's stable sort."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 1023, 1024, 1025, 5000, 7169, 8191, 8192, 8193])
@pytest.mark.parametrize("end_bit", [1, 8, 9, 17, 40, 64])
def test_sorts_of_one_block(n, end_bit):
    from paper_2411_06224_gb300 import binding as B

    ctx = B.gs_create(0)
    rng = np.random.default_rng(n + end_bit)
    keys = rng.integers(0, 2**63, n, dtype=np.uint64) << np.uint64(1) | rng.integers(0, 2, n, dtype=np.uint64)
    if n % 2:  # many equal keys
        keys = keys[rng.integers(0, max(n // 7, 1), n)]
    vals = rng.integers(0, 2**31, n).astype(np.int32)
    ko, vo = B.gs_prim_sort_pairs(ctx, torch.as_tensor(keys.view(np.int64), device="cuda"), torch.as_tensor(vals, device="cuda"), end_bit)
    order = np.argsort(keys & np.uint64((1 << end_bit) - 1), kind="stable")
    assert np.array_equal(vo.cpu().numpy(), vals[order])
    assert np.array_equal(ko.cpu().numpy().view(np.uint64), keys[order])
    B.gs_destroy(ctx)
