"""Assembly of matrices with rows of more than 4,096 inputs beside short ones: keys bit
for bit, sums within 1e-13 of the sum of magnitudes, the input map, and the short
rows' bits, which do not depend on another row's length."""

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


def dev(a, dt):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def assemble(B, ctx, n, rows, cols, blocks):
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    out = [v.cpu().numpy() for v in B.gs_mat_export(ctx, mat)]
    B.gs_mat_destroy(mat)
    return out


def scene(n, lens, seed, shuffle):
    """Row i of lens[i] inputs on random columns (many of them twice), and inputs below the diagonal."""
    rng = np.random.default_rng(seed)
    rows = np.concatenate([np.full(l, i) for i, l in lens.items()])
    cols = rows + (rng.integers(0, n, rows.size) % (n - rows))
    low = rng.integers(1, n, 300)
    rows, cols = np.concatenate([rows, low]), np.concatenate([cols, low - 1])
    if shuffle:
        p = rng.permutation(rows.size)
        rows, cols = rows[p], cols[p]
    return rows, cols, rng.normal(size=(rows.size, 3, 3))


CASES = [(40, {0: 4097, 3: 10, 39: 4096}), (40, {5: 70_001, 6: 1, 7: 33, 8: 5000, 38: 4500, 39: 9000}),
         (50_000, {0: 200_000, 1: 7, 49_999: 4100, 100: 256, 20_000: 4097}),
         (3000, {i: 4097 + 3 * i for i in range(0, 300, 7)} | {i: 5 for i in range(1000, 2000)}), (1, {0: 30_000})]


@pytest.mark.parametrize("n,lens", CASES)
@pytest.mark.parametrize("shuffle", [False, True])
def test_long_rows_beside_short_ones(B, ctx, n, lens, shuffle):
    rows, cols, blocks = scene(n, lens, n + len(lens), shuffle) if n > 1 else (
        np.zeros(30_000, int), np.zeros(30_000, int), np.random.default_rng(1).normal(size=(30_000, 3, 3)))
    rid, cid, au = assemble(B, ctx, n, rows, cols, blocks)
    keep = rows <= cols
    key, inv = np.unique(rows[keep].astype(np.int64) * n + cols[keep], return_inverse=True)
    assert np.array_equal(rid.astype(np.int64) * n + cid, key)
    want, mag = np.zeros((key.size, 9)), np.zeros((key.size, 9))
    np.add.at(want, inv, blocks[keep].reshape(-1, 9))
    np.add.at(mag, inv, np.abs(blocks[keep].reshape(-1, 9)))
    assert (np.abs(au.reshape(-1, 9) - want) <= 1e-13 * mag).all()
    # the rows of up to 4,096 inputs alone
    count = np.bincount(rows[keep], minlength=n)
    short = count[rows] <= 4096
    if short.any():
        r2, c2, a2 = assemble(B, ctx, n, rows[short], cols[short], blocks[short])
        at = count[rid] <= 4096
        assert np.array_equal(rid[at], r2) and np.array_equal(cid[at], c2) and np.array_equal(au[at], a2)


def test_input_map_of_long_rows(B, ctx):
    rng = np.random.default_rng(9)
    n, hubs = 6000, 3
    i = np.arange(n)
    rows, cols, blocks = [i], [i], [np.repeat(4.0 * np.eye(3)[None], n, 0)]
    blocks[0][:hubs] *= 2 * n
    for h in range(hubs):
        c = rng.integers(h + 1, n, 5000 + h)
        rows.append(np.full(c.size, h)), cols.append(c), blocks.append(rng.uniform(-0.3, 0.3, (c.size, 3, 3)) / hubs)
    rows.append(np.array([5, 9])), cols.append(np.array([2, 1])), blocks.append(np.ones((2, 3, 3)))  # not consumed
    rows, cols, blocks = (np.concatenate(v) for v in (rows, cols, blocks))
    p = rng.permutation(rows.size)
    rows, cols, blocks = rows[p], cols[p], blocks[p]
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(i, torch.int32), (n + 31) // 32, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=32, max_levels=1)
    rid, cid, _ = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    x, g = dev(rng.normal(size=(1, 3 * n)), torch.float64), dev(rng.normal(size=(1, 3 * n)), torch.float64)
    dH = torch.empty((rid.size, 3, 3), dtype=torch.float64, device="cuda")
    dI = torch.full((rows.size, 3, 3), 7.0, dtype=torch.float64, device="cuda")
    B.gs_adjoint(ctx, mat, m, x, g, dLdH=dH, dLdinput=dI)
    at = np.searchsorted(rid.astype(np.int64) * n + cid, rows.astype(np.int64) * n + cols)
    keep = rows <= cols
    want = np.where(keep[:, None, None], dH.cpu().numpy()[np.minimum(at, rid.size - 1)], 0.0)
    assert np.array_equal(dI.cpu().numpy(), want)
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
