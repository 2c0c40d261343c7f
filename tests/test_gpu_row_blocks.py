"""Rows that the warps of a block sum together: lengths at its edges, runs that span
several warps' pieces (one column, two, a few, all different), and the numeric assembly
of a fan of tets, which sums by the same rule.

Tolerance: sums of at most n values in any order agree to n 2^-53 of the sum of
magnitudes; 1e-12 covers 4,096 and, in the fans, the elements' own 1e-13.
"""

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


def summed(n, rows, cols, blocks):
    keep = rows <= cols
    key, inv = np.unique(rows[keep].astype(np.int64) * n + cols[keep], return_inverse=True)
    want, mag = np.zeros((key.size, 9)), np.zeros((key.size, 9))
    np.add.at(want, inv, blocks[keep].reshape(-1, 9))
    np.add.at(mag, inv, np.abs(blocks[keep].reshape(-1, 9)))
    return key, want, mag


@pytest.mark.parametrize("columns", [1, 2, 5, 40, 3000])
def test_rows_of_a_block(B, ctx, columns):
    rng = np.random.default_rng(columns)
    lens = [255, 256, 257, 258, 271, 272, 273, 511, 512, 513, 1000, 2047, 2048, 2049, 4081, 4095, 4096, 1]
    n = len(lens) + columns
    rows = np.concatenate([np.full(l, i) for i, l in enumerate(lens)])
    cols = len(lens) + rng.integers(0, columns, rows.size)
    for i, l in enumerate(lens):  # the diagonal too: a run of a third of the row
        at = np.nonzero(rows == i)[0]
        cols[at[: l // 3]] = i
    p = rng.permutation(rows.size)
    rows, cols, blocks = rows[p], cols[p], rng.normal(size=(rows.size, 3, 3))
    out = []
    for _ in range(2):
        mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
        out.append([v.cpu().numpy() for v in B.gs_mat_export(ctx, mat)])
        B.gs_mat_destroy(mat)
    key, want, mag = summed(n, rows, cols, blocks)
    rid, cid, au = out[0]
    assert np.array_equal(rid.astype(np.int64) * n + cid, key)
    assert (np.abs(au.reshape(-1, 9) - want) <= 1e-12 * mag).all()
    assert np.array_equal(au, out[1][2])  # a fixed order


@pytest.mark.parametrize("T", [60, 64, 65, 128, 500, 1000, 1023, 1100, 30_000])
def test_numeric_assembly_of_a_fan(B, ctx, T):
    rng = np.random.default_rng(T)
    X = np.concatenate([np.zeros((1, 3)), rng.normal(size=(3 * T, 3)) + [3.0, 0.0, 0.0]])
    tets = np.stack([np.zeros(T, int), *(1 + np.arange(3 * T).reshape(T, 3).T)], 1)
    d = X[tets[:, 1:]] - X[tets[:, :1]]
    flip = np.einsum("ij,ij->i", d[:, 0], np.cross(d[:, 1], d[:, 2])) < 0
    tets[flip, 1], tets[flip, 2] = tets[flip, 2].copy(), tets[flip, 1].copy()
    fem = B.gs_fem_create(ctx, dev(X, torch.float64), dev(tets, torch.int32), 1e5, 0.4, 1000.0, 0.01)
    x = dev(X + 0.01 * rng.normal(size=X.shape), torch.float64)
    t = B.gs_fem_triplets(ctx, fem, x, 10 * T + X.shape[0])
    mat, ref = B.gs_fem_assemble(ctx, fem, x), B.gs_assemble(ctx, X.shape[0], *t)
    a, b = ([v.cpu().numpy() for v in B.gs_mat_export(ctx, m)] for m in (mat, ref))
    key, want, mag = summed(X.shape[0], *(v.cpu().numpy() for v in t))
    for rid, cid, au in (a, b):
        assert np.array_equal(rid.astype(np.int64) * X.shape[0] + cid, key)
        assert (np.abs(au.reshape(-1, 9) - want) <= 1e-12 * mag).all()
    if 4 * T <= 4000:  # no row of more than 4,096 inputs: the same sums in the same order
        assert np.array_equal(a[2], b[2])
    B.gs_mat_destroy(mat)
    B.gs_mat_destroy(ref)
    B.gs_fem_destroy(fem)
