"""Assembly with rows sorted one by one: rows at the edges of the warp and
block sorts (1, 32, 33, 64, 65, 128, 129, 256 inputs; 257, 512, 513, 4,096 for
a block), one input more (the general path), empty rows, inputs below the
diagonal, and few inputs on many rows (general path).  Keys bit for bit, sums
against 1e-13 of the sum of magnitudes, and the input map through the adjoint's
gather."""

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


def check(B, ctx, n, rows, cols, blocks):
    t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    mat = B.gs_assemble(ctx, n, t(rows, torch.int32), t(cols, torch.int32), t(blocks, torch.float64))
    rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    B.gs_mat_destroy(mat)
    keep = rows <= cols
    key, inv = np.unique(rows[keep].astype(np.int64) * n + cols[keep], return_inverse=True)
    assert np.array_equal(rid, key // n) and np.array_equal(cid, key % n)
    want, mag = np.zeros((key.size, 9)), np.zeros((key.size, 9))
    np.add.at(want, inv, blocks[keep].reshape(-1, 9))
    np.add.at(mag, inv, np.abs(blocks[keep].reshape(-1, 9)))
    assert (np.abs(au.reshape(-1, 9) - want) <= 1e-13 * mag).all()


@pytest.mark.parametrize("longest", [256, 4096, 4097])
def test_row_lengths(B, ctx, longest):
    rng = np.random.default_rng(longest)
    lens = [l for l in (0, 1, 2, 31, 32, 33, 0, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1025, 4095)
            if l <= longest] + [longest, 0]
    n = 60
    rows = np.concatenate([np.full(l, 2 * i) for i, l in enumerate(lens)])
    cols = rows + (rng.integers(0, n, rows.size) % (n - rows))  # many duplicates
    low = rng.integers(1, n, 500)  # below the diagonal: not consumed
    rows, cols = np.concatenate([rows, low]), np.concatenate([cols, low - 1])
    perm = rng.permutation(rows.size)
    check(B, ctx, n, rows[perm].astype(np.int32), cols[perm].astype(np.int32), rng.normal(size=(rows.size, 3, 3)))


@pytest.mark.parametrize("n,nb", [(1, 1), (1, 5000), (7, 3), (400_000, 50), (3, 40)])
def test_sizes(B, ctx, n, nb):
    rng = np.random.default_rng(n + nb)
    r, c = rng.integers(0, n, nb), rng.integers(0, n, nb)
    check(B, ctx, n, r.astype(np.int32), c.astype(np.int32), rng.normal(size=(nb, 3, 3)))


def test_only_lower_inputs(B, ctx):
    r = np.arange(1, 50, dtype=np.int32)
    check(B, ctx, 50, r, r - 1, np.ones((r.size, 3, 3)))


def test_refill_with_a_vertex_of_thousands_of_tets(B, ctx):
    """Numeric assembly where runs are longer than a window, and longer than the
    split into windows allows: a fan of tets around one vertex, against numpy sums
    of the same triplets."""
    rng = np.random.default_rng(5)
    for T in (40, 300, 1100, 5000):
        X = np.concatenate([np.zeros((1, 3)), rng.normal(size=(3 * T, 3)) + [3.0, 0.0, 0.0]])
        tets = np.stack([np.zeros(T, int), *(1 + np.arange(3 * T).reshape(T, 3).T)], 1)
        d = X[tets[:, 1:]] - X[tets[:, :1]]
        flip = np.einsum("ij,ij->i", d[:, 0], np.cross(d[:, 1], d[:, 2])) < 0
        tets[flip, 1], tets[flip, 2] = tets[flip, 2].copy(), tets[flip, 1].copy()
        t = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
        fem = B.gs_fem_create(ctx, t(X, torch.float64), t(tets, torch.int32), 1e5, 0.4, 1000.0, 0.01)
        x = t(X + 0.01 * rng.normal(size=X.shape), torch.float64)
        rows, cols, blocks = B.gs_fem_triplets(ctx, fem, x, 10 * T + X.shape[0])
        mat = B.gs_fem_assemble(ctx, fem, x)
        rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
        key, inv = np.unique(rows.cpu().numpy().astype(np.int64) * X.shape[0] + cols.cpu().numpy(), return_inverse=True)
        want, mag = np.zeros((key.size, 9)), np.zeros((key.size, 9))
        np.add.at(want, inv, blocks.cpu().numpy().reshape(-1, 9))
        np.add.at(mag, inv, np.abs(blocks.cpu().numpy().reshape(-1, 9)))
        assert np.array_equal(rid.astype(np.int64) * X.shape[0] + cid, key)
        assert (np.abs(au.reshape(-1, 9) - want) <= 1e-12 * mag).all()
        B.gs_mat_destroy(mat)
        B.gs_fem_destroy(fem)
