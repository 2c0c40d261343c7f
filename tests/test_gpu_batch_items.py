"""Batched PCG where its work items can go wrong: empty and one-node systems, sizes
on both sides of an item's and of a quarter item's end, in a graph and out of it.

Chains of 3 x 3 blocks (4.5 I on the diagonal plus a rank-one part, -I off it).
Tolerance: a solve to 1e-6 stops on the recurrence's residual, which parts from
the true one by rounding alone, here far below 5 % of 1e-6.
"""

import numpy as np
import pytest
import torch

from oracle import pcg

pytestmark = pytest.mark.gpu

SIZES = [1, 0, 2, 85, 86, 341, 342, 0, 1365, 1366, 3001, 1, 0]


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


@pytest.mark.parametrize("chunk", [1024, 4096])
@pytest.mark.parametrize("use_graph", [True, False])
@pytest.mark.parametrize("prec,tc", [(0, 4), (0, 0), (1, 4)])  # the forms with and without separate products
def test_ragged_systems_reach_the_residual_asked_for(B, ctx, chunk, use_graph, prec, tc):
    rng = np.random.default_rng(5)
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int32)
    n = int(off[-1])
    last = np.zeros(n, dtype=bool)
    last[off[1:][np.array(SIZES) > 0] - 1] = True
    i = np.arange(n, dtype=np.int32)
    e = i[~last]  # chain edges (e, e + 1) within a system
    u = rng.normal(size=(n, 3))
    diag = 4.5 * np.eye(3) + u[:, :, None] * u[:, None, :]
    rows = np.concatenate([i, e]).astype(np.int32)
    cols = np.concatenate([i, e + 1]).astype(np.int32)
    blocks = np.concatenate([diag, np.repeat(-np.eye(3)[None], len(e), 0)])
    deg = np.zeros(n, dtype=np.int64)
    np.add.at(deg, e, 1)
    np.add.at(deg, e + 1, 1)
    ptr = np.concatenate([[0], np.cumsum(deg)])
    adj = np.concatenate([[j for j in (k - 1, k + 1) if 0 <= j < n and not last[min(j, k)]] for k in range(n)])
    B.gs_tune_set(ctx, B.GS_TUNE_BATCH_CHUNK, chunk)
    B.gs_tune_set(ctx, B.GS_TUNE_F64_TC, tc)
    try:
        mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
        X = np.stack([i, np.zeros(n), np.zeros(n)], 1).astype(np.float64)
        mp, nd = B.gs_partition_batch(X, off, 16)
        m = B.gs_build_mas(ctx, mat, dev(mp, torch.int32), nd, dev(ptr, torch.int32), dev(adj, torch.int32), None,
                           domain_size=16, max_levels=3, precision=prec)
        b = rng.normal(size=3 * n)
        b[3 * off[4] : 3 * off[5]] = 0.0
        x = torch.full((3 * n,), 7.0, dtype=torch.float64, device="cuda")
        it, rel, _ = B.gs_pcg_solve_batch(ctx, mat, m, off, dev(b, torch.float64), x, tol=1e-6, use_graph=use_graph)
        xg = x.cpu().numpy()
        # the assembly keeps every key once: the lists above are the sorted matrix's entries
        res = b - pcg.spmv(rows, cols, blocks, xg.reshape(-1, 3)).ravel()
        for s in range(len(SIZES)):
            sl = slice(3 * off[s], 3 * off[s + 1])
            if not b[sl].any():
                assert it[s] == 0 and not xg[sl].any()
            else:
                assert it[s] >= 1 and rel[s] <= 1e-6
                assert np.linalg.norm(res[sl]) <= 1.05e-6 * np.linalg.norm(b[sl])
        it, rel, st = B.gs_pcg_solve_batch(ctx, mat, m, off, dev(b, torch.float64), x, tol=1e-6, max_iter=2,
                                           use_graph=use_graph, raise_on_maxiter=False)
        assert st == B.GS_ERR_MAXITER and int(np.max(it)) == 2
        B.gs_mas_destroy(m)
        B.gs_mat_destroy(mat)
    finally:
        B.gs_tune_set(ctx, B.GS_TUNE_BATCH_CHUNK, 4096)
        B.gs_tune_set(ctx, B.GS_TUNE_F64_TC, 4)
