"""Device bisection against the host rule where its lists and slot kernels can
go wrong: parts longer than a warp (slots by sorting), single vertices, ties
and negative zeros in the coordinates, and bodies of very different size."""

import numpy as np
import pytest
import torch

from synth.mesh import adjacency_csr

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


@pytest.mark.parametrize("n,N", [(1, 1), (1, 32), (2, 1), (31, 32), (33, 32), (1000, 31), (1000, 33), (1000, 48),
                                 (5000, 700), (777, 1000)])
def test_bisection_matches_host(B, ctx, n, N):
    X = np.round(np.random.default_rng(n + N).normal(size=(n, 3)) * 4) / 4  # many equal coordinates
    X[np.random.default_rng(1).random(X.shape) < 0.1] = -0.0
    mp, nd = B.gs_partition(X, N)
    md, ndd = B.gs_partition_device(ctx, torch.as_tensor(X, device="cuda"), N)
    assert nd == ndd
    assert np.array_equal(mp, md.cpu().numpy())


@pytest.mark.parametrize("N", [4, 32, 40])
def test_components_match_host_per_body(B, ctx, N):
    """Each body is bisected on its own, bodies numbered by their smallest vertex."""
    rng = np.random.default_rng(N)
    sizes = [1, 3000, 2, 130, 1, 700]
    n = sum(sizes)
    body = rng.permutation(np.repeat(np.arange(len(sizes)), sizes))
    X = rng.normal(size=(n, 3))
    edges = np.concatenate([np.stack([v[:-1], v[1:]], 1) for b in range(len(sizes))
                            for v in [np.nonzero(body == b)[0]] if v.size > 1])
    ptr, adj = adjacency_csr(n, edges)
    md, nd = B.gs_partition_device(ctx, torch.as_tensor(X, device="cuda"), N, rule=B.GS_PART_RCB_COMPONENTS,
                                   adj_ptr=torch.as_tensor(ptr, device="cuda"), adj=torch.as_tensor(adj, device="cuda"))
    want, parts = np.empty(n, np.int32), 0
    for b in sorted(range(len(sizes)), key=lambda q: np.nonzero(body == q)[0][0]):
        v = np.nonzero(body == b)[0]
        m, k = B.gs_partition(X[v], N)
        want[v] = m + parts * N
        parts += k
    assert nd == parts
    assert np.array_equal(want, md.cpu().numpy())
