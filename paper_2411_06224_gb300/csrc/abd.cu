// Two-level reduction for coupled FEM / affine-body Hessians (Sec. 5.1, Sec. 5.2).
//
// Level 1 reduces every 3x3 contact / element block per full-space node
// pair (r, c) with the FastHashReduction of assemble.cu.  Each unique pair
// is then mapped once through the Jacobians: with w(i) = [1, xbar_i] for a
// body node (x_i = A xbar_i + p, q = [p; a_1; a_2; a_3]) the product
// J_r^T C J_c consists of the 3x3 sub-blocks w_a(r) w_b(c) C, which are
// emitted on the reduced block rows (16 for body-body, 4 for body-FEM, 1
// for FEM-FEM: Sec. 5.2's unification), and level 2 reduces them again.
// Both orientations (r, c, C) and (c, r, C^T) of an off-diagonal pair are
// expanded so that every reduced sub-block lands in the upper triangle.
// Indices n_nodes + 4b + a name body b's own reduced block row a directly:
// a body's 12 x 12 Hessian (inertia, orthogonality potential) enters as its
// 16 sub-blocks, Sec. 5.2's ABD-ABD block type, and passes level 2 with
// weight 1.

#include "common.cuh"
#include "primitives.cuh"
#include "sort_scan.cuh"

namespace gs {

int reduce_blocks(gs_ctx ctx, int32_t n, const int32_t* rows, const int32_t* cols, const double* blocks,
                  int64_t nb, gs_mat* out);

struct AbdMap {
  const int32_t* body;
  const double* xbar;
  int32_t n_fem;
  int32_t n_bodies;
  int32_t n_nodes;
};

__device__ __forceinline__ int abd_targets(const AbdMap& m, int32_t node, int32_t* R, double* w) {
  if (node >= m.n_nodes) {  // a body's own reduced block row (its 12 x 12 Hessian's 3 x 3 sub-blocks)
    R[0] = m.n_fem + (node - m.n_nodes);
    w[0] = 1.0;
    return 1;
  }
  int32_t b = m.body[node];
  if (b < 0) {
    R[0] = node;
    w[0] = 1.0;
    return 1;
  }
  int32_t base = m.n_fem + 4 * b;
  R[0] = base;
  R[1] = base + 1;
  R[2] = base + 2;
  R[3] = base + 3;
  w[0] = 1.0;
  w[1] = m.xbar[3 * node + 0];
  w[2] = m.xbar[3 * node + 1];
  w[3] = m.xbar[3 * node + 2];
  return 4;
}

__global__ void k_abd_validate(AbdMap m, int32_t n_nodes, int* flags) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  int32_t b = m.body[i];
  bool ok = (b < 0) ? (i < m.n_fem) : (b < m.n_bodies && i >= m.n_fem);
  if (!ok) atomicOr(flags, kErrIndex);
}

// Sub-blocks that each stored pair emits: orientation (r, c), then (c, r) of an
// off-diagonal pair, (a, b) ascending, those on or above the diagonal.
__global__ void k_abd_count(AbdMap m, const int32_t* __restrict__ rid, const int32_t* __restrict__ cid, int64_t U,
                            int32_t* __restrict__ cnt) {
  int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u >= U) return;
  const int32_t r = rid[u], c = cid[u];
  int32_t Rr[4], Rc[4];
  double wr[4], wc[4];
  const int nr = abd_targets(m, r, Rr, wr), nc = abd_targets(m, c, Rc, wc);
  int count = 0;
  for (int orient = 0; orient < (r == c ? 1 : 2); ++orient)
    for (int a = 0; a < (orient ? nc : nr); ++a)
      for (int b = 0; b < (orient ? nr : nc); ++b) count += (orient ? Rc[a] : Rr[a]) <= (orient ? Rr[b] : Rc[b]);
  cnt[u] = count;
}

// Emits them, a warp per 32 pairs.  What bounds it: the bytes written, so a warp
// writes whole runs: pairs of single rows (most) are copied, nine neighbouring
// lanes a block; any other pair is taken by the whole warp, lane 16 orient + 4 a
// + b deciding on one sub-block and its weight, then the lanes along the
// values.  A thread per pair, writing its sub-blocks value by value, took 201 us
// for the 40^3 body with 1000 affine cubes, this 57.
constexpr int kAbdWarps = 8;
__global__ void __launch_bounds__(32 * kAbdWarps) k_abd_emit(AbdMap m, const int32_t* __restrict__ rid,
                                                             const int32_t* __restrict__ cid,
                                                             const double* __restrict__ au, int64_t U,
                                                             const int32_t* __restrict__ off,
                                                             int32_t* __restrict__ orow, int32_t* __restrict__ ocol,
                                                             double* __restrict__ oblk) {
  __shared__ double s_w[kAbdWarps][2][32][3];  // weights 1..3 of each pair's row and column
  __shared__ double s_scale[kAbdWarps][32], s_C[kAbdWarps][9];
  __shared__ int s_trans[kAbdWarps][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t u0 = ((int64_t)blockIdx.x * kAbdWarps + wid) * 32, u = u0 + lane;
  if (u0 >= U) return;  // whole warp
  int32_t Rr[4] = {0, 0, 0, 0}, Rc[4] = {0, 0, 0, 0};
  int nr = 0, nc = 0;
  int32_t at = 0, r = 0, c = 0;
  if (u < U) {
    double wr[4], wc[4];
    r = rid[u], c = cid[u], at = off[u];
    nr = abd_targets(m, r, Rr, wr), nc = abd_targets(m, c, Rc, wc);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (nr == 4) s_w[wid][0][lane][k] = wr[k + 1];
      if (nc == 4) s_w[wid][1][lane][k] = wc[k + 1];
    }
  }
  // single rows both (r < c or r == c): one block, weight 1
  const bool single = nr == 1 && nc == 1 && Rr[0] <= Rc[0] && (r == c || Rc[0] > Rr[0]);
  const uint32_t singles = __ballot_sync(kFull, single), others = __ballot_sync(kFull, nr > 0 && !single);
  if (single) orow[at] = Rr[0], ocol[at] = Rc[0];
  __syncwarp();
  if (singles)
#pragma unroll
    for (int t = lane; t < 32 * 9; t += 32) {
      const int i = t / 9;
      const int32_t to = __shfl_sync(kFull, at, i);
      if ((singles >> i) & 1u) oblk[(int64_t)to * 9 + (t - 9 * i)] = au[u0 * 9 + t];
    }
  for (uint32_t left = others; left; left &= left - 1) {
    const int i = __ffs(left) - 1;
    const int na_ = __shfl_sync(kFull, nr, i), nb_ = __shfl_sync(kFull, nc, i);
    const int32_t R0 = __shfl_sync(kFull, Rr[0], i), C0 = __shfl_sync(kFull, Rc[0], i);
    const bool diag = __shfl_sync(kFull, r, i) == __shfl_sync(kFull, c, i);
    const int32_t o = __shfl_sync(kFull, at, i);
    const int orient = lane >> 4, a = (lane >> 2) & 3, b = lane & 3;
    const int32_t RA = (orient ? C0 : R0) + a, RB = (orient ? R0 : C0) + b;  // a body's rows are consecutive
    const bool emit = a < (orient ? nb_ : na_) && b < (orient ? na_ : nb_) && RA <= RB && !(orient && diag);
    const uint32_t em = __ballot_sync(kFull, emit);
    const int rank = __popc(em & ((1u << lane) - 1u));
    if (emit) {
      const double wa = a ? s_w[wid][orient][i][a - 1] : 1.0, wb = b ? s_w[wid][orient ^ 1][i][b - 1] : 1.0;
      s_scale[wid][rank] = wa * wb;
      s_trans[wid][rank] = orient;
      orow[o + rank] = RA;
      ocol[o + rank] = RB;
    }
    if (lane < 9) s_C[wid][lane] = au[(u0 + i) * 9 + lane];
    __syncwarp();
    const int values = 9 * __popc(em);
    for (int t = lane; t < values; t += 32) {
      const int k = t / 9, q = t - 9 * k;
      oblk[(int64_t)o * 9 + t] = s_scale[wid][k] * s_C[wid][s_trans[wid][k] ? 3 * (q % 3) + q / 3 : q];
    }
    __syncwarp();
  }
}

}  // namespace gs

using namespace gs;

extern "C" int gs_assemble_abd(gs_ctx ctx, int32_t n_nodes, int32_t n_fem, int32_t n_bodies,
                               const int32_t* body_of_node, const double* xbar, const int32_t* rows,
                               const int32_t* cols, const double* blocks, int64_t n_blocks, gs_mat* out) {
  GS_CHECK(ctx && out, GS_ERR_INVALID, "gs_assemble_abd: null context or output");
  *out = nullptr;
  GS_CHECK(n_nodes > 0 && n_fem >= 0 && n_fem <= n_nodes && n_bodies >= 0, GS_ERR_INVALID,
           "gs_assemble_abd: bad sizes");
  GS_CHECK(body_of_node && (n_bodies == 0 || xbar), GS_ERR_INVALID, "gs_assemble_abd: null body map");
  int64_t n_red = (int64_t)n_fem + 4LL * n_bodies;
  GS_CHECK(n_red > 0 && n_red < (1 << 30), GS_ERR_INVALID, "gs_assemble_abd: reduced size out of range");
  GS_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  AbdMap m{body_of_node, xbar, n_fem, n_bodies, n_nodes};
  { GS_PROF(ctx, GS_K_OTHER); k_abd_validate<<<ceil_div(n_nodes, 256), 256, 0, st>>>(m, n_nodes, ctx->d_flags); }
  int flags = 0;
  GS_TRY(ctx->take_flags(&flags));
  if (flags) return status_from_flags(flags);
  gs_mat lvl1 = nullptr;
  GS_CHECK((int64_t)n_nodes + 4LL * n_bodies < (1LL << 30), GS_ERR_INVALID, "gs_assemble_abd: too many rows");
  GS_TRY(gs_assemble(ctx, n_nodes + 4 * n_bodies, rows, cols, blocks, n_blocks, &lvl1));
  int64_t U = lvl1->nnzb;
  int32_t *cnt = nullptr, *off = nullptr, *orow = nullptr, *ocol = nullptr;
  double* oblk = nullptr;
  void* temp = nullptr;
  size_t tb = 0;
  int s = GS_OK;
  int64_t total = 0;
  if ((s = ctx->alloc((void**)&cnt, (size_t)(U + 1) * 4)) || (s = ctx->alloc((void**)&off, (size_t)(U + 1) * 4)))
    goto done;
  if (U > 0) {
    { GS_PROF(ctx, GS_K_ASSEMBLE); k_abd_count<<<ceil_div(U, 256), 256, 0, st>>>(m, lvl1->rid, lvl1->cid, U, cnt); }
  }
  cudaMemsetAsync(cnt + U, 0, 4, st);
  tb = scan_temp_bytes(U + 1);
  if ((s = ctx->alloc(&temp, tb))) goto done;
  {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    if ((s = exclusive_scan_i32(st, cnt, off, U + 1, temp, tb))) goto done;
  }
  if (cudaMemcpyAsync(ctx->h_pinned, off + U, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess) {
    set_error("gs_assemble_abd: readback failed");
    s = GS_ERR_CUDA;
    goto done;
  }
  total = ctx->h_pinned[0];
  if ((s = ctx->alloc((void**)&orow, (size_t)total * 4)) || (s = ctx->alloc((void**)&ocol, (size_t)total * 4)) ||
      (s = ctx->alloc((void**)&oblk, (size_t)total * 72)))
    goto done;
  if (U > 0) {
    { GS_PROF(ctx, GS_K_ASSEMBLE); k_abd_emit<<<ceil_div(U, 32 * kAbdWarps), 32 * kAbdWarps, 0, st>>>(m, lvl1->rid, lvl1->cid, lvl1->au, U, off, orow,
                                                                       ocol, oblk); }
  }
  s = gs_assemble(ctx, (int32_t)n_red, orow, ocol, oblk, total, out);
done:
  ctx->release(cnt);
  ctx->release(off);
  ctx->release(temp);
  ctx->release(orow);
  ctx->release(ocol);
  ctx->release(oblk);
  gs_mat_destroy(lvl1);
  return s;
}
