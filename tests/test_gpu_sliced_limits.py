"""PCG on matrices whose sliced copy would be mostly padding (one row coupled to very
many nodes): the product runs over the stored matrix then, to the same end.

Tolerance: a solve to 1e-6 stops on the recurrence's residual, which parts from
the true one by rounding alone, here (about ten iterations) far below 5 % of 1e-6.
"""

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


@pytest.mark.parametrize("n,hubs", [(3000, 1), (70_000, 1), (70_000, 40)])  # sliced; one slice of padding; hubs fill theirs
@pytest.mark.parametrize("nrhs", [1, 4])
@pytest.mark.parametrize("ff", [False, True])
def test_rows_coupled_to_every_node(B, ctx, n, hubs, nrhs, ff):
    rng = np.random.default_rng(n + hubs)
    i = np.arange(n, dtype=np.int32)
    rows, cols = [i], [i]
    blocks = [np.repeat(4.0 * np.eye(3)[None], n, 0)]
    blocks[0][:hubs] *= n
    for h in range(hubs):
        c = np.arange(h + 1, n, dtype=np.int32)
        if hubs > 1:
            c = c[rng.random(len(c)) < 0.5]
        rows.append(np.full(len(c), h, np.int32)), cols.append(c)
        blocks.append(rng.uniform(-0.5, 0.5, (len(c), 3, 3)) / hubs)
    rows, cols, blocks = np.concatenate(rows), np.concatenate(cols), np.concatenate(blocks)
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(i, torch.int32), (n + 31) // 32, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=32, max_levels=1)
    b = rng.normal(size=(nrhs, 3 * n))
    x = torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
    for _ in range(2):
        it, rel, _ = B.gs_pcg_solve(ctx, mat, m, dev(b, torch.float64), x, nrhs=nrhs, tol=1e-6,
                                    variant=B.GS_SPMV_ROW_FF if ff else B.GS_SPMV_ROW)
        xg = x.cpu().numpy()
        for q in range(nrhs):
            Ax = pcg.spmv(rows, cols, blocks, xg[q].reshape(-1, 3)).ravel()
            assert np.linalg.norm(b[q] - Ax) <= 1.05e-6 * np.linalg.norm(b[q]) and rel[q] <= 1e-6
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
