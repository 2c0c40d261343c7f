"""GS_TUNE_F64_TC 1, 2 and 4 are one form of the FP64 preconditioner: solves launch the
same kernels with each and give the same bits (every reduction has a fixed order), and
the autotuner does not choose among them by noise."""

import numpy as np
import pytest
import torch

from synth.workloads import make_tet_system, rhs, uneven_batch

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


def build(B, ctx, s, N, node_off=None):
    mat = B.gs_assemble(ctx, s.n_vertices, dev(s.rows, torch.int32), dev(s.cols, torch.int32), dev(s.blocks, torch.float64))
    mp, nd = B.gs_partition(s.X, N) if node_off is None else B.gs_partition_batch(s.X, node_off, N)
    M = B.gs_build_mas(ctx, mat, dev(mp, torch.int32), nd, dev(s.adj_ptr, torch.int32), dev(s.adj, torch.int32),
                       dev(s.contacts, torch.int32), domain_size=N, max_levels=3)
    return mat, M


def each_value(B, ctx, run):
    """{value: (launches per kernel class, result)}"""
    out = {}
    try:
        for tc in (4, 1, 2):
            B.gs_tune_set(ctx, B.GS_TUNE_F64_TC, tc)
            run()  # the copies that a matrix makes on its first solve
            B.gs_profile_begin(ctx, [])
            res = run()
            out[tc] = list(B.gs_profile_end(ctx)[0]), res
    finally:
        B.gs_tune_set(ctx, B.GS_TUNE_F64_TC, 4)
    return out


def same(out):
    for tc in (1, 2):
        assert out[tc][0] == out[4][0], (tc, out[tc][0], out[4][0])
        assert torch.equal(out[tc][1], out[4][1]), tc


@pytest.mark.parametrize("cells,N,nrhs", [(9, 32, 1), (9, 16, 3), (13, 32, 8)])
def test_solves_do_not_depend_on_the_value(B, ctx, cells, N, nrhs):
    s = make_tet_system(cells, E=1e6, n_contacts=3 * cells, contact_mode="near", seed=cells)
    mat, M = build(B, ctx, s, N)
    b = dev(rhs(3 * s.n_vertices, nrhs), torch.float64)

    def run():
        x = torch.zeros_like(b)
        B.gs_pcg_solve(ctx, mat, M, b, x, nrhs=nrhs, tol=1e-6)
        return x

    same(each_value(B, ctx, run))
    from paper_2411_06224_gb300 import autotune

    times = autotune.tune(ctx, mat, M, nrhs=nrhs, reps=2, fp64=True)["fp64_on_tensor_cores"][1]
    for p in autotune.CANDIDATES:  # the defaults again
        B.gs_tune_set(ctx, p, {B.GS_TUNE_SPMV_LANES: 2, B.GS_TUNE_APPLY_RHS: 4, B.GS_TUNE_SPMV32_LANES: 2,
                               B.GS_TUNE_BATCH_CHUNK: 4096, B.GS_TUNE_BF16_TC: 1, B.GS_TUNE_F64_TC: 4,
                               B.GS_TUNE_SPMV_WINDOW: 1024, B.GS_TUNE_SPMV_WS: 1, B.GS_TUNE_SPMV_FF_RHS: 8}[p])
    assert set(times) == {4, 0}
    B.gs_mas_destroy(M)
    B.gs_mat_destroy(mat)


def test_batches_do_not_depend_on_the_value(B, ctx):
    bt = uneven_batch(n_sys=4, v_range=(300, 3000), e_range=(1e5, 1e7), seed=5)
    mat, M = build(B, ctx, bt, 32, node_off=bt.node_off)
    b = dev(rhs(3 * bt.n_vertices, 1)[0], torch.float64)

    def run():
        x = torch.zeros_like(b)
        B.gs_pcg_solve_batch(ctx, mat, M, bt.node_off, b, x, tol=1e-6)
        return x

    same(each_value(B, ctx, run))
    B.gs_mas_destroy(M)
    B.gs_mat_destroy(mat)
