"""The digit bytes of the FP64 tensor-core apply where a row's leading digit is at
its limits: inverses whose largest entries lie just below a power of two, on both
sides of 127.498 / 128, from which the row takes one exponent more, and powers of
two themselves.

Diagonal systems: z = v r with v the inverse's entry.  Tolerance, of |v r|: the
inverse is within 4 ulp of v (one square root, one division and one product);
the digits keep 2^-54 of the row's largest entry, which is v, and of the
right-hand side's largest, which is at most 4 |r| here; dropped digit products
are below 2^-55 of both; the result is rounded once.  Together below
4 2^-52 + 2^-54 + 4 2^-54 + 4 2^-55 + 2^-53 < 2^-49.
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


@pytest.mark.parametrize("N", [16, 32])
@pytest.mark.parametrize("domains", [1, 3, 400, 1300])  # per SM: one at most, two, more
@pytest.mark.parametrize("nrhs", [1, 4, 5, 8])
def test_rows_at_the_leading_digits_limits(B, ctx, N, domains, nrhs):
    n = N * domains - 5  # the last domain is ragged
    rng = np.random.default_rng(n + nrhs)
    edge = np.array([1.0, 1.0 + 2.0**-52, 1.5, 2.0 - 2.0**-52, 2.0 - 2.0**-20, 2.0 * 127.5 / 128, 2.0 * 127.498 / 128,
                     2.0 * 127.498046875 / 128, 2.0 * 127.4980 / 128, 2.0 * 127.4 / 128, 1.9921, 1.99219, 1.992187])
    v = edge[rng.integers(0, len(edge), 3 * n)] * 2.0 ** rng.integers(-30, 30, 3 * n)
    idx = np.arange(n, dtype=np.int32)
    blocks = np.zeros((n, 3, 3))
    for c in range(3):
        blocks[:, c, c] = 1.0 / v[c::3]
    mat = B.gs_assemble(ctx, n, dev(idx, torch.int32), dev(idx, torch.int32), dev(blocks, torch.float64))
    m = B.gs_build_mas(ctx, mat, dev(idx, torch.int32), domains, dev(np.zeros(n + 1), torch.int32),
                       dev(np.zeros(1), torch.int32), None, domain_size=N, max_levels=1)
    r = rng.uniform(0.25, 1.0, (nrhs, 3 * n)) * rng.choice([-1.0, 1.0], (nrhs, 3 * n))
    z = torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
    B.gs_mas_apply(ctx, m, dev(r, torch.float64), z, nrhs=nrhs)
    err = np.abs(z.cpu().numpy() - v * r) / np.abs(v * r)
    assert err.max() <= 2.0**-49
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
