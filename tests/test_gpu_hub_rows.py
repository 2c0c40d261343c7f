"""PCG on large systems with one row coupled to a few hundred nodes, on both sides of
the length from which four lanes share every row, by the true residual (a solve to 1e-6
stops on the recurrence's, which parts from it by far less than 5 % here)."""

import numpy as np
import pytest
import torch

from oracle import pcg

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


@pytest.mark.parametrize("entries", [192, 193, 1000])
@pytest.mark.parametrize("nrhs", [1, 3, 8])
@pytest.mark.parametrize("ff", [False, True])
def test_rows_of_many_entries(B, ctx, entries, nrhs, ff):
    n = 90_000
    rng = np.random.default_rng(entries)
    i = np.arange(n, dtype=np.int32)
    c = np.sort(rng.choice(np.arange(1, n), entries - 1, replace=False)).astype(np.int32)
    rows, cols = np.concatenate([i, i[:-1], np.zeros_like(c)]), np.concatenate([i, i[1:], c])
    blocks = np.concatenate([np.repeat(4.0 * np.eye(3)[None], n, 0), rng.uniform(-0.4, 0.4, (n - 1, 3, 3)),
                             rng.uniform(-0.5, 0.5, (c.size, 3, 3))])
    blocks[0] *= entries
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(i, torch.int32), (n + 31) // 32, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=32, max_levels=1)
    rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    b = rng.normal(size=(nrhs, 3 * n))
    x = torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
    _, rel, _ = B.gs_pcg_solve(ctx, mat, m, dev(b, torch.float64), x, nrhs=nrhs, tol=1e-6,
                               variant=B.GS_SPMV_ROW_FF if ff else B.GS_SPMV_ROW)
    xg = x.cpu().numpy()
    for q in range(nrhs):
        Ax = pcg.spmv(rid, cid, au, xg[q].reshape(-1, 3)).ravel()
        assert np.linalg.norm(b[q] - Ax) <= 1.05e-6 * np.linalg.norm(b[q]) and rel[q] <= 1e-6
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
