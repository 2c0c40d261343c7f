"""W^T W on the tensor cores: domain inverses of every number of real nodes, and of
matrices whose rows differ by many powers of two.

A = D B D with B = I + small symmetric part (eigenvalues in [0.5, 1.5]) and D powers
of two, so A^-1 = D^-1 B^-1 D^-1 exactly; Cholesky, the inverse factor and W^T W
all commute with D.  Tolerance, entry by entry of D A^-1 D: 3 products of 96 terms
on a matrix of condition 3, 3 x 96 x 2^-53 x 3 plus the digits' 2^-54 x 16, below
2^-42.
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


@pytest.mark.parametrize("N", [16, 32, 24, 8])  # 24 and 8: the product in FP64
@pytest.mark.parametrize("spread", [0, 8, 40])
@pytest.mark.parametrize("prec", [0, 1])
def test_inverses_of_every_size(B, ctx, N, spread, prec):
    rng = np.random.default_rng(N + spread)
    sizes = list(range(1, N + 1))  # domain d has d + 1 real nodes
    n, nd = sum(sizes), len(sizes)
    slot = np.concatenate([N * d + rng.permutation(N)[:k] for d, k in enumerate(sizes)]).astype(np.int32)
    D = 2.0 ** rng.integers(-spread, spread + 1, 3 * n)
    rows, cols, blocks, want = [], [], [], []
    for d, k in enumerate(sizes):
        o = sum(sizes[:d])
        S = rng.normal(size=(3 * k, 3 * k))
        S = (S + S.T) / np.linalg.norm(S + S.T, 2) * 0.5 + np.eye(3 * k)
        want.append(np.linalg.inv(S))
        s = D[3 * o : 3 * (o + k)]
        A = s[:, None] * S * s[None, :]
        for a in range(k):
            for b in range(a, k):
                rows.append(o + a), cols.append(o + b), blocks.append(A[3 * a : 3 * a + 3, 3 * b : 3 * b + 3])
    mat = B.gs_assemble(ctx, n, dev(rows, torch.int32), dev(cols, torch.int32), dev(np.array(blocks), torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(slot, torch.int32), nd, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=N, max_levels=1, precision=prec)
    inv = B.gs_mas_export_inverse(ctx, m, 0, nd, N).cpu().numpy()
    tol = 2.0**-42 if prec == 0 else 2.0**-22  # FP32: the stored inverse is rounded
    for d, k in enumerate(sizes):
        o = sum(sizes[:d])
        at = np.concatenate([3 * (slot[o : o + k] - N * d)[:, None] + np.arange(3)]).reshape(-1)
        s = D[3 * o : 3 * (o + k)]
        got = s[:, None] * inv[d][np.ix_(at, at)] * s[None, :]
        assert np.abs(got - want[d]).max() <= tol, (d, np.abs(got - want[d]).max())
        pad = np.ones(3 * N, dtype=bool)
        pad[at] = False
        assert np.all(inv[d][pad] == 0) and np.all(inv[d][:, pad] == 0)
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
