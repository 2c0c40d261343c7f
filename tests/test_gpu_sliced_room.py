"""PCG where the device has little room left: the sliced copy of the matrix is optional,
so a solve succeeds wherever its vectors and scalars fit, whatever part of the copy
would fit beside them, and gives the same solution.

The room is a memory pool of a fixed size that the device allocates from for the time
of the solve (matrix, row order and preconditioner are older), swept from little more than
the solve itself needs (14 MB, and the pool's own granularity) to more than the whole copy (0.13 GB), finely where the copy
just fits and only what is allocated after it could fail.
"""

import ctypes

import numpy as np
import pytest
import torch

from oracle import pcg

pytestmark = pytest.mark.gpu

MB = 1 << 20


class Location(ctypes.Structure):
    _fields_ = [("type", ctypes.c_int), ("id", ctypes.c_int)]


class PoolProps(ctypes.Structure):  # CUmemPoolProps
    _fields_ = [("allocType", ctypes.c_int), ("handleTypes", ctypes.c_int), ("location", Location),
                ("win32", ctypes.c_void_p), ("maxSize", ctypes.c_size_t), ("usage", ctypes.c_ushort),
                ("reserved", ctypes.c_ubyte * 54)]


@pytest.fixture(scope="module")
def B():
    from paper_2411_06224_gb300.build import build

    build()
    from paper_2411_06224_gb300 import binding

    return binding


def system(n):
    """Rows coupled to the next 13 nodes: 27 blocks each in the full matrix."""
    rng = np.random.default_rng(3)
    i = np.arange(n, dtype=np.int32)
    rows = np.concatenate([i] + [i[:-k] for k in range(1, 14)])
    cols = np.concatenate([i] + [i[k:] for k in range(1, 14)])
    blocks = rng.uniform(-0.05, 0.05, (rows.size, 3, 3))
    blocks[:n] = 3.0 * np.eye(3)
    return rows, cols, blocks


def test_solves_fit_where_their_vectors_fit(B):
    cuda = ctypes.CDLL("libcuda.so.1")

    def check(status):
        assert status == 0, status

    torch.cuda.init()
    torch.zeros(1, device="cuda")
    n, nrhs = 60_000, 2
    rows, cols, blocks = system(n)
    d = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    i = np.arange(n, dtype=np.int32)
    trip = d(rows, torch.int32), d(cols, torch.int32), d(blocks, torch.float64)
    levels = (d(i, torch.int32), (n + 31) // 32, d(np.zeros(n + 1), torch.int32), d(np.zeros(1), torch.int32), None)
    b = np.random.default_rng(4).normal(size=(nrhs, 3 * n))
    bd, x = d(b, torch.float64), torch.empty((nrhs, 3 * n), dtype=torch.float64, device="cuda")
    copy = 27 * n * 80 / MB  # 124
    sizes = [48, 64, 96, 112] + list(range(int(copy) + 4, int(copy) + 40)) + [224, 320]
    default = ctypes.c_void_p()
    check(cuda.cuDeviceGetDefaultMemPool(ctypes.byref(default), 0))
    for mb in sizes:
        ctx = B.gs_create(0)
        mat = B.gs_assemble(ctx, n, *trip)
        m = B.gs_build_mas(ctx, mat, *levels, domain_size=32, max_levels=1)
        B.gs_spmv(ctx, mat, bd, x, nrhs=nrhs, variant=B.GS_SPMV_ROW)  # what the product needs in any case
        torch.cuda.synchronize()
        pool = ctypes.c_void_p()
        check(cuda.cuMemPoolCreate(ctypes.byref(pool), ctypes.byref(PoolProps(1, 0, Location(1, 0), None, mb * MB, 0))))
        check(cuda.cuDeviceSetMemPool(0, pool))
        try:
            for _ in range(2):
                x.zero_()
                _, rel, _ = B.gs_pcg_solve(ctx, mat, m, bd, x, nrhs=nrhs, tol=1e-8, variant=B.GS_SPMV_ROW)
                assert (np.array(rel) <= 1e-8).all(), mb
        finally:
            check(cuda.cuDeviceSetMemPool(0, default))
            B.gs_mas_destroy(m)
            B.gs_mat_destroy(mat)
            B.gs_destroy(ctx)
            check(cuda.cuMemPoolDestroy(pool))
        xg = x.cpu().numpy()
        for q in range(nrhs):
            r = b[q] - pcg.spmv(rows, cols, blocks, xg[q].reshape(-1, 3)).ravel()
            assert np.linalg.norm(r) <= 1.05e-8 * np.linalg.norm(b[q]), mb
