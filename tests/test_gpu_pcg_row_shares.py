"""PCG's FP64 product of 3, 5, 6 and 7 right-hand sides on both sides of the sizes (for
152 SMs) at which the lanes of a row and the threads of a block change: the residual that
PCG reports against the one on the host, and the iterations against one right-hand side's
(a wrong p . Ap of any would cost the A-orthogonality, and with it iterations)."""

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


def dev(a, dt):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("n", [38_912, 38_913, 116_737, 155_648, 155_649, 233_473, 466_945])
def test_shares_of_the_row_product(B, n):
    ctx = B.gs_create(0)
    rng = np.random.default_rng(n)
    i = np.arange(n, dtype=np.int32)
    far = np.minimum(i + rng.integers(2, 60, n), n - 1).astype(np.int32)
    rows = np.concatenate([i, i[:-1], i[far > i]])
    cols = np.concatenate([i, i[1:], far[far > i]])
    off = rng.uniform(-0.3, 0.3, (rows.size - n, 3, 3))
    blocks = np.concatenate([np.repeat(5.0 * np.eye(3)[None], n, 0), off])
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(i, torch.int32), (n + 31) // 32, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=32, max_levels=1, precision=B.GS_PREC_FP32)
    rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    b = rng.normal(size=(7, 3 * n))
    one = None
    for nrhs in (1, 3, 5, 6, 7):
        x = torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
        it, rel, _ = B.gs_pcg_solve(ctx, mat, m, dev(b[:nrhs], torch.float64), x, nrhs=nrhs, tol=1e-6,
                                    variant=B.GS_SPMV_ROW)
        xg = x.cpu().numpy()
        one = int(it[0]) if one is None else one
        assert all(abs(int(k) - one) <= 2 for k in it), (nrhs, it)  # the same matrix, random right-hand sides
        for q in range(nrhs):
            Ax = pcg.spmv(rid, cid, au, xg[q].reshape(-1, 3)).ravel()
            assert np.linalg.norm(b[q] - Ax) <= 1.05e-6 * np.linalg.norm(b[q]) and rel[q] <= 1e-6, (nrhs, q)
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
    B.gs_destroy(ctx)
