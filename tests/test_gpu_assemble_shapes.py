"""Assembly on both sides of the sizes at which its kernels change: few rows with many
inputs each (counted in shared memory; all rows sorted together), many rows with few
(the general path), rows of 1,024 and 1,025 inputs (8 or 32 warps).  Keys bit for bit,
sums within 1e-13 of the sum of magnitudes (at most 10^3 inputs to a block on average),
and an index out of range is still refused."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2411_06224_gb300.build import build

    build()
    from paper_2411_06224_gb300 import binding

    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.gs_create(0)
    yield c
    B.gs_destroy(c)


def check(B, ctx, n, rows, cols):
    blocks = np.random.default_rng(n).normal(size=(rows.size, 3, 3))
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    mat = B.gs_assemble(ctx, n, t(rows, torch.int32), t(cols, torch.int32), t(blocks, torch.float64))
    rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    B.gs_mat_destroy(mat)
    keep = rows <= cols
    key, inv = np.unique(rows[keep].astype(np.int64) * n + cols[keep], return_inverse=True)
    assert np.array_equal(rid.astype(np.int64) * n + cid, key)
    want, mag = np.zeros((key.size, 9)), np.zeros((key.size, 9))
    for q in range(9):
        v = blocks[keep].reshape(-1, 9)[:, q]
        want[:, q], mag[:, q] = np.bincount(inv, v, key.size), np.bincount(inv, np.abs(v), key.size)
    assert (np.abs(au.reshape(-1, 9) - want) <= 1e-13 * mag).all()


# n, inputs: few rows (256 inputs per row and 16,384 inputs; 8,192 rows), together (2,304 and 4,096 inputs per row,
# 256 and 1,024 rows, 8 rows and 400,000 inputs), many rows (400,000; three inputs per row)
CASES = [(63, 16_383), (63, 16_384), (64, 16_383), (65, 16_640), (100, 25_599), (8192, 8192 * 256), (8193, 8193 * 256),
         (255, 255 * 2304 - 1), (255, 255 * 2304), (256, 256 * 2304), (8, 399_999), (8, 400_000), (9, 400_000),
         (1023, 1023 * 4096), (400_000, 10_000), (400_001, 10_000), (400_001, 1_200_003), (400_001, 1_200_002)]


@pytest.mark.parametrize("n,nb", CASES)
def test_sizes_where_the_kernels_change(B, ctx, n, nb):
    rng = np.random.default_rng(n + nb)
    rows = rng.integers(0, n, nb)
    check(B, ctx, n, rows, np.clip(rows + rng.integers(-1, 40, nb), 0, n - 1))


@pytest.mark.parametrize("length", [1024, 1025])
def test_rows_of_eight_and_of_thirty_two_warps(B, ctx, length):
    rng = np.random.default_rng(length)
    rows = np.repeat(np.arange(0, 60, 3), length)
    rows = np.concatenate([rows, rng.integers(0, 60, 500)])
    check(B, ctx, 60, rows, np.minimum(rows + rng.integers(0, 7, rows.size), 59))


def test_few_rows_refuse_bad_indices(B, ctx):
    for bad in (-1, 50):
        r = np.random.default_rng(1).integers(0, 50, 20_000)
        r[12_345] = bad
        t = torch.as_tensor(r.astype(np.int32), device="cuda")
        b = torch.zeros((r.size, 3, 3), dtype=torch.float64, device="cuda")
        with pytest.raises(B.GsError):
            B.gs_assemble(ctx, 50, t, t, b)
        with pytest.raises(B.GsError):
            B.gs_assemble(ctx, 50, torch.zeros_like(t), t, b)
