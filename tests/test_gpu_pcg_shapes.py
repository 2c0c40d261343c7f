"""PCG's iteration kernels at every shape they are built for, by the true residual.

Right-hand sides 1..9 (9 takes the separate passes), levels 1..4, domains of
16, 24 and 32, FP64 and FP32 preconditioners, both row products, node counts off
every tile, more domains than one reduction holds partial sums for, systems on
both sides of the size from which the kernels are launched singly, and a solve
that stops at its first iteration.

Tolerance: a solve to 1e-6 stops on the recurrence's residual, which parts from
the true one by rounding alone: at most a few hundred iterations x 2^-47 x the
condition number of the scaled steps, below 5 % of 1e-6 (the margin that the
oracle comparison of the solver uses as well).
"""

import numpy as np
import pytest
import torch

from oracle import assembly, pcg
from synth.workloads import make_tet_system, rhs

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


_SYS = {}


def system(cells):
    if cells not in _SYS:
        _SYS.clear()  # the cases are ordered by size
        s = make_tet_system(cells, E=1e6, n_contacts=3 * cells, contact_mode="near", seed=cells)
        _SYS[cells] = (s, *assembly.assemble(s.rows, s.cols, s.blocks))
    return _SYS[cells]


# cells, domain size, levels, precision (0 FP64, 1 FP32), right-hand sides, product (0 row, 2 float-float)
CASES = [(5, 32, 1, 0, 1, 0), (5, 16, 2, 0, 2, 2), (5, 24, 2, 0, 3, 0), (5, 32, 2, 1, 1, 2),
         (7, 16, 4, 0, 5, 2), (7, 32, 3, 1, 8, 0), (7, 24, 3, 1, 2, 2), (7, 32, 2, 0, 9, 0), (7, 32, 2, 0, 9, 2),
         (11, 32, 3, 0, 1, 2), (11, 32, 3, 0, 8, 2), (11, 16, 3, 1, 3, 0), (11, 32, 4, 0, 4, 0),
         (26, 16, 3, 0, 1, 0), (26, 16, 3, 1, 4, 2), (42, 32, 3, 0, 8, 2), (42, 32, 3, 1, 8, 0)]


@pytest.mark.parametrize("cells,N,L,prec,nrhs,variant", CASES)
def test_solution_has_the_residual_asked_for(B, ctx, cells, N, L, prec, nrhs, variant):
    s, rid, cid, au = system(cells)
    V = s.n_vertices
    variant = {0: B.GS_SPMV_ROW, 2: B.GS_SPMV_ROW_FF}[variant]
    mat = B.gs_assemble(ctx, V, dev(s.rows, torch.int32), dev(s.cols, torch.int32), dev(s.blocks, torch.float64))
    map_, ndom = B.gs_partition(s.X, N)
    m = B.gs_build_mas(ctx, mat, dev(map_, torch.int32), ndom, dev(s.adj_ptr, torch.int32), dev(s.adj, torch.int32),
                       dev(s.contacts, torch.int32), domain_size=N, max_levels=L,
                       precision=B.GS_PREC_FP32 if prec else B.GS_PREC_FP64)
    b = rhs(3 * V, nrhs)
    if nrhs > 2:
        b[nrhs - 1] = 0.0  # stops before the first iteration; the others go on
    x = torch.full((nrhs, 3 * V), 7.0, dtype=torch.float64, device="cuda")
    it, rel, _ = B.gs_pcg_solve(ctx, mat, m, dev(b, torch.float64), x, nrhs=nrhs, tol=1e-6, variant=variant)
    xg = x.cpu().numpy()
    for q in range(nrhs):
        if not b[q].any():
            assert it[q] == 0 and not xg[q].any()
            continue
        Ax = pcg.spmv(rid, cid, au, xg[q].reshape(-1, 3)).ravel()
        assert rel[q] <= 1e-6 and it[q] > 1
        assert np.linalg.norm(b[q] - Ax) <= 1.05e-6 * np.linalg.norm(b[q])
    # one iteration, then the cap: the residual that is reported is that of x
    it, rel, st = B.gs_pcg_solve(ctx, mat, m, dev(b, torch.float64), x, nrhs=nrhs, tol=1e-6, max_iter=1,
                                 variant=variant, raise_on_maxiter=False)
    xg = x.cpu().numpy()
    assert st == B.GS_ERR_MAXITER
    for q in range(nrhs):
        if b[q].any():
            Ax = pcg.spmv(rid, cid, au, xg[q].reshape(-1, 3)).ravel()
            true = np.linalg.norm(b[q] - Ax) / np.linalg.norm(b[q])
            assert it[q] == 1 and abs(true - rel[q]) <= 1e-9 * max(true, 1.0)
    B.gs_mas_destroy(m)
    B.gs_mat_destroy(mat)
