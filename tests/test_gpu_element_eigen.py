"""Element Hessians where the 3x3 eigenproblems have no gaps or small ones: rest,
rotations, equal and nearly equal stretches, inversions, flattened tets, and noise
from 1e-15 to 1e-1 on each.

Tolerance: both sides are backward stable and the projection onto the PSD cone is
1-Lipschitz, so an element's blocks agree to a few hundred ulps of its largest
entry whatever the gaps (eigenvectors of a near-degenerate pair may turn within
their plane; the projected block does not depend on it): 1e-11, as in the
element-by-element comparison of a deformed body.
"""

import numpy as np
import pytest
import torch

from oracle import elastic

pytestmark = pytest.mark.gpu

NU, RHO, DT = 0.4, 1000.0, 0.01


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


STRETCHES = [(1, 1, 1), (0.5, 0.5, 0.5), (1.7, 1.7, 1.7), (1, 1, 1.3), (0.8, 1.2, 1.2), (1, 1 + 1e-8, 1 + 2e-8),
             (1, 1 + 1e-4, 1.5), (0.1, 1, 3), (1, 1, -1), (0.7, 0.7, -0.7), (0.9, 1.1, -1e-3), (1, 1, 0), (0.3, 0.6, 0.9)]


@pytest.mark.parametrize("noise", [0.0, 1e-15, 1e-12, 1e-9, 1e-7, 1e-5, 1e-3, 1e-1])
@pytest.mark.parametrize("E", [1.0, 1e5, 1e12])
def test_projected_blocks_without_gaps(B, ctx, noise, E):
    rng = np.random.default_rng(3)
    X0 = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1.0]]) * 0.01
    X, x = [], []
    for k, s in enumerate(STRETCHES * 5):
        q1, q2 = (np.linalg.qr(rng.normal(size=(3, 3)))[0] for _ in range(2))
        q1, q2 = q1 * np.linalg.det(q1), q2 * np.linalg.det(q2)
        F = np.diag(s) if k < len(STRETCHES) else q1 @ np.diag(s) @ q2.T
        F = F + noise * rng.normal(size=(3, 3))
        X.append(X0 + 0.05 * k)
        x.append(X0 @ F.T + rng.normal(size=3))
    X, x = np.concatenate(X), np.concatenate(x)
    T = len(X) // 4
    tets = np.arange(4 * T, dtype=np.int32).reshape(T, 4)
    f = B.gs_fem_create(ctx, dev(X), dev(tets, torch.int32), E, NU, RHO, DT)
    _, _, b = B.gs_fem_triplets(ctx, f, dev(x), 10 * T + 4 * T)
    b = b.cpu().numpy()[: 10 * T].reshape(T, 10, 3, 3)
    H = elastic.element_hessians(X, x, tets, E, NU).reshape(T, 4, 3, 4, 3)
    pairs = [(i, j) for i in range(4) for j in range(i, 4)]
    want = np.stack([H[:, i, :, j, :] for i, j in pairs], 1)
    # positions lie up to 4 from the origin and F is their difference over 0.01: its
    # own rounding is 400 ulps on both sides, the same inputs and another order
    scale = np.abs(want).reshape(T, -1).max(axis=1)
    err = np.abs(b - want).reshape(T, -1).max(axis=1)
    assert np.all(err <= 1e-11 * scale), (err / scale).max()
    B.gs_fem_destroy(f)
