"""Element Hessians around the uniform stretch at which two eigenvalues of the 3x3
block vanish together (mu = lam (s^3 - alpha) s): one may be slightly positive and
the other slightly negative while every leading minor rounds to a positive number.

Tolerance: unit tets, so F carries a few ulps on both sides, both projections are
backward stable to some hundred ulps and the projection is 1-Lipschitz: entries agree
to 1e-12 of the element's largest, and a symmetric 12 x 12 matrix within that of a
positive semi-definite one has no eigenvalue below -12 times it.
"""

import numpy as np
import pytest
import torch

from oracle import elastic

pytestmark = pytest.mark.gpu

RHO, DT = 1000.0, 0.01


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


def dev(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("nu", [0.3, 0.4, 0.49])
@pytest.mark.parametrize("E", [1.0, 1e6])
def test_blocks_near_the_double_root_are_projected(B, ctx, nu, E):
    rng = np.random.default_rng(int(100 * nu))
    mu, lam = elastic.lame(E, nu)
    alpha = 1.0 + mu / lam
    s0 = max(r.real for r in np.roots([lam, 0.0, 0.0, -lam * alpha, -mu]) if abs(r.imag) < 1e-9)
    T = 4000
    e = 10.0 ** rng.uniform(-11, -5, T)
    X0 = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1.0]])
    X = np.tile(X0, (T, 1))
    q = np.linalg.qr(rng.normal(size=(2, T, 3, 3)))[0]
    q *= np.linalg.det(q)[..., None, None]
    F = q[0] @ (s0 * (1.0 + e[:, None] * rng.normal(size=(T, 3)))[:, :, None] * q[1])
    x = np.einsum("ai,tji->taj", X0, F).reshape(-1, 3)
    tets = np.arange(4 * T, dtype=np.int32).reshape(T, 4)
    f = B.gs_fem_create(ctx, dev(X), dev(tets, torch.int32), E, nu, RHO, DT)
    _, _, b = B.gs_fem_triplets(ctx, f, dev(x), 10 * T + 4 * T)
    b = b.cpu().numpy()[: 10 * T].reshape(T, 10, 3, 3)
    H = np.empty((T, 4, 3, 4, 3))
    for p, (i, j) in enumerate((i, j) for i in range(4) for j in range(i, 4)):
        H[:, i, :, j, :] = b[:, p]
        H[:, j, :, i, :] = b[:, p].transpose(0, 2, 1)
    H = H.reshape(T, 12, 12)
    H = 0.5 * (H + H.transpose(0, 2, 1))
    want = elastic.element_hessians(X, x, tets, E, nu).reshape(T, 12, 12)
    scale = np.abs(want).reshape(T, -1).max(axis=1)
    low = np.linalg.eigvalsh(H)[:, 0] / scale
    assert low.min() >= -12e-12, low.min()
    err = np.abs(H - want).reshape(T, -1).max(axis=1) / scale
    assert err.max() <= 1e-12, err.max()
    B.gs_fem_destroy(f)
