"""The expansion of affine-body pairs where a warp's 32 pairs mix kinds: single rows,
body-vertex, body-body (the same body and two), a body's own rows, in counts off
a warp's and a block's size.

Every value is one product of two weights and a block entry, summed per key; the
oracle sums the same terms in another order, so entries agree to the number of
terms of a key times 2^-52 times the sum of their magnitudes: 64 terms at most
here, checked as 2^-45 of the largest magnitude per block times the terms.
"""

import numpy as np
import pytest
import torch

from oracle import assembly

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


@pytest.mark.parametrize("n_fem,bodies,pairs", [(1, 1, 1), (5, 0, 31), (0, 2, 33), (40, 3, 255), (40, 3, 257),
                                                (300, 20, 3000)])
def test_mixed_pairs_match_the_oracle(B, ctx, n_fem, bodies, pairs):
    rng = np.random.default_rng(100 * n_fem + bodies)
    n_nodes = n_fem + 8 * bodies
    body = np.concatenate([np.full(n_fem, -1), np.repeat(np.arange(bodies), 8)]).astype(np.int32)
    xbar = rng.normal(size=(n_nodes, 3))
    r, c = rng.integers(0, n_nodes, pairs), rng.integers(0, n_nodes, pairs)
    r, c = np.minimum(r, c).astype(np.int32), np.maximum(r, c).astype(np.int32)
    blocks = rng.normal(size=(pairs, 3, 3))
    sym = r == c
    blocks[sym] += blocks[sym].transpose(0, 2, 1)
    # every diagonal entry, so that no row is empty
    r = np.concatenate([r, np.arange(n_nodes)]).astype(np.int32)
    c = np.concatenate([c, np.arange(n_nodes)]).astype(np.int32)
    blocks = np.concatenate([blocks, np.repeat(np.eye(3)[None], n_nodes, 0)])
    mat = B.gs_assemble_abd(ctx, n_nodes, n_fem, bodies, dev(body, torch.int32), dev(xbar, torch.float64),
                            dev(r, torch.int32), dev(c, torch.int32), dev(blocks, torch.float64))
    rid, cid, au = B.gs_mat_export(ctx, mat)
    oid, ocid, oau = assembly.assemble_abd(r, c, blocks, body, xbar, n_fem)
    assert np.array_equal(rid.cpu().numpy(), oid) and np.array_equal(cid.cpu().numpy(), ocid)
    _, _, mag = assembly.assemble_abd(r, c, np.abs(blocks), body, np.abs(xbar), n_fem)
    assert np.all(np.abs(au.cpu().numpy() - oau) <= 2.0**-45 * mag.max(axis=(1, 2), keepdims=True))
    B.gs_mat_destroy(mat)
