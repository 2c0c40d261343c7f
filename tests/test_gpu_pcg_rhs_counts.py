"""PCG's product for every number of right-hand sides up to 8 on both sides of the sizes
at which lanes share them differently, by the true residual (a solve to 1e-6 stops on
the recurrence's, which parts from it by far less than 5 %), and a right-hand side's
iterations, which do not depend on how many others there are."""

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


@pytest.mark.parametrize("n", [500, 4095, 4096, 50_001, 100_000])
@pytest.mark.parametrize("ff", [False, True])
@pytest.mark.parametrize("prec", [0, 1])
def test_every_number_of_right_hand_sides(B, ctx, n, ff, prec):
    rng = np.random.default_rng(n)
    i = np.arange(n, dtype=np.int32)
    far = np.minimum(i + rng.integers(2, 60, n), n - 1).astype(np.int32)
    rows = np.concatenate([i, i[:-1], i[far > i]])
    cols = np.concatenate([i, i[1:], far[far > i]])
    off = rng.uniform(-0.3, 0.3, (rows.size - n, 3, 3))
    blocks = np.concatenate([np.repeat(5.0 * np.eye(3)[None], n, 0), off])
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(i, torch.int32), (n + 31) // 32, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=32, max_levels=1,
                       precision=B.GS_PREC_FP32 if prec else B.GS_PREC_FP64)
    rid, cid, au = (v.cpu().numpy() for v in B.gs_mat_export(ctx, mat))
    b = rng.normal(size=(8, 3 * n))
    variant = B.GS_SPMV_ROW_FF if ff else B.GS_SPMV_ROW
    alone = None
    for nrhs in range(1, 9):
        x = torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
        it, rel, _ = B.gs_pcg_solve(ctx, mat, m, dev(b[:nrhs], torch.float64), x, nrhs=nrhs, tol=1e-6, variant=variant)
        xg = x.cpu().numpy()
        alone = it[0] if alone is None else alone
        assert abs(int(it[0]) - int(alone)) <= 1
        for q in range(nrhs):
            Ax = pcg.spmv(rid, cid, au, xg[q].reshape(-1, 3)).ravel()
            assert np.linalg.norm(b[q] - Ax) <= 1.05e-6 * np.linalg.norm(b[q]) and rel[q] <= 1e-6, (nrhs, q)
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
