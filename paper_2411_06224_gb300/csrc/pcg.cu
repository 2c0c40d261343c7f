// Preconditioned conjugate gradients for several right-hand sides (Sec. 3.2).
//
// Per iteration (one SpMV per RHS):
//   Ap = A p, alpha = rz / (p . Ap)
//   x += alpha p, r -= alpha Ap, ||r||^2 and the per-RHS convergence test
//   z = M^{-1} r, beta = (r . z) / rz, rz = r . z
//   p = z + beta p
// For up to 8 right-hand sides each line but the third is one kernel
// (pcg_fused.cu), and where the preconditioner's form allows it (mas_dot_usable)
// the second also restricts r and the third also takes r . z: five kernels,
// launched so that each is resident when the one before it ends.  Other counts
// and forms run the product, the dot product or the apply as separate passes
// (k_dot, k_update_xr here).
// Every reduction is deterministic: a fixed grid writes partial sums, and the
// kernels that need the scalar add them in a fixed order (pcg_state.cuh), so
// no scalar ever travels to the host inside the loop.  The convergence test of
// an iteration is taken with its direction update.  A RHS stops moving once
// converged (alpha = 0), which keeps each RHS on exactly its own single-RHS
// recurrence.  Kernels return at once after every RHS converged; the host polls
// that flag every four iterations, one poll behind, so that the GPU always has
// the next iterations queued.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "ff.cuh"
#include "pcg_state.cuh"
#include "primitives.cuh"

namespace gs {

int spmv_launch(gs_ctx ctx, gs_mat m, const double* x, double* y, int nrhs, int variant);
int mas_apply_launch(gs_ctx ctx, gs_mas mas, const double* r, double* z, int nrhs, double* rl, double* zl);
int mas_level_vectors(gs_ctx ctx, gs_mas mas, int nrhs, double** rl, double** zl);
int ensure_row_order(gs_ctx ctx, gs_mat m);

int pcg_spmv_dot(gs_ctx ctx, gs_mat m, const float2* ps, const double* p, double* Ap, int nrhs, const PcgScalars* s,
                 Partials& pap);
int pcg_update_xr(gs_ctx ctx, gs_mas mas, double* x, double* r, const double* p, const double* Ap, int nrhs, double* rl,
                  int64_t lstride, PcgScalars* s, const Partials& pap, Partials& rrp, int parity);
int pcg_update_p(gs_ctx ctx, gs_mat m, double* p, const double* z, float2* ps, int nrhs, PcgScalars* s,
                 const Partials& rrp, const Partials& rzp, Partials fold, double tol2, int parity);
bool mas_dot_usable(gs_ctx ctx, gs_mas mas, int nrhs);
int mas_products(gs_ctx ctx, gs_mas mas, const double* r, double* z, int nrhs, double* rl, double* zl, const int* skip,
                 const Partials* dot);

constexpr int kRedThreads = 256;
constexpr int kMaxChunks = 256;     // reduction blocks per right-hand side of the kernels here
constexpr int kUnroll = 4;          // strided elements per thread and pass of k_dot

// Grid of the vector kernels: (G, nrhs); block (g, k) covers a contiguous
// chunk of right-hand side k.  G depends only on the vector length, the RHS
// count and the GPU's SM count, so on one GPU the reduction order -- and
// therefore the result -- is fixed.
inline int red_blocks(int64_t len, int nrhs, int sms) {
  // 32 entries per thread: each block's reduction, fence and arrival are
  // fixed costs, so blocks are made long (measured: 8 per thread left k_dot
  // stalled on its block reductions at 21 % of the DRAM peak) -- but no
  // fewer than about two blocks per SM over all RHS while a block still gets
  // 8 entries per thread
  int64_t g = (len + kRedThreads * 32 - 1) / (kRedThreads * 32);
  const int64_t want = (2LL * std::max(sms, 1) + nrhs - 1) / nrhs;
  const int64_t cap8 = (len + kRedThreads * 8 - 1) / (kRedThreads * 8);
  g = std::max(g, std::min(want, cap8));
  return (int)std::max<int64_t>(1, std::min<int64_t>(g, kMaxChunks));
}

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red[kRedThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x < 32) {
    t = threadIdx.x < kRedThreads / 32 ? red[threadIdx.x] : 0.0;
    t = warp_sum(t);
  }
  __syncthreads();
  return t;  // valid in warp 0
}

__device__ __forceinline__ int block_max(int v) {
  __shared__ int red[kRedThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(kFull, v, o));
  if (lane == 0) red[w] = v;
  __syncthreads();
  int t = kExpNone;
  if (threadIdx.x < 32) {
    t = threadIdx.x < kRedThreads / 32 ? red[threadIdx.x] : kExpNone;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t = max(t, __shfl_xor_sync(kFull, t, o));
  }
  __syncthreads();
  return t;  // valid in warp 0
}

__device__ __forceinline__ void chunk_of(int64_t len, int64_t& b, int64_t& e) {
  const int64_t per = (len + gridDim.x - 1) / gridDim.x;
  b = (int64_t)blockIdx.x * per;
  e = b + per < len ? b + per : len;
}

// Partial sums of a_k . b_k, block (g, k) its chunk of right-hand side k; kCopy
// also writes dst = b (p = z); kEx also the exponent bound of the chunk of b
// (z) for the float-float SpMV operand.
template <bool kCopy, bool kEx>
__global__ void __launch_bounds__(kRedThreads) k_dot(const double* __restrict__ a, const double* __restrict__ b,
                                                     double* __restrict__ dst, int64_t len, const int* __restrict__ skip,
                                                     Partials out) {
  if (skip && *skip) return;
  const int64_t o = (int64_t)blockIdx.y * len;
  int64_t i0, i1;
  chunk_of(len, i0, i1);
  // kUnroll strided elements per pass, loaded before they are summed: more
  // loads in flight per thread, and the thread's sum keeps its order
  double v = 0.0;
  int ex = kExpNone;
  const int64_t T = blockDim.x;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += kUnroll * T) {
    double av[kUnroll], bv[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t j = i + u * T;
      av[u] = j < i1 ? a[o + j] : 0.0;
      bv[u] = j < i1 ? b[o + j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t j = i + u * T;
      if (j < i1) {
        v += av[u] * bv[u];
        if (kCopy) dst[o + j] = bv[u];
        if (kEx) ex = max(ex, ex_bound(bv[u]));
      }
    }
  }
  v = block_sum(v);
  if (kEx) ex = block_max(ex);
  if (threadIdx.x == 0) {
    out.sum[blockIdx.y * out.pitch + blockIdx.x] = v;
    if (kEx) out.ex[blockIdx.y * out.pitch + blockIdx.x] = ex;
  }
}

// x = 0, r = b, partial sums of ||b||^2.
__global__ void __launch_bounds__(kRedThreads) k_init(const double* __restrict__ bvec, double* __restrict__ x,
                                                      double* __restrict__ r, int64_t len, Partials out) {
  const int64_t o = (int64_t)blockIdx.y * len;
  int64_t i0, i1;
  chunk_of(len, i0, i1);
  double v = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const double bb = bvec[o + i];
    x[o + i] = 0.0;
    r[o + i] = bb;
    v += bb * bb;
  }
  v = block_sum(v);
  if (threadIdx.x == 0) out.sum[blockIdx.y * out.pitch + blockIdx.x] = v;
}

// The first scalars, block k right-hand side k (s is zeroed): ||b||^2, rz = r . z
// of the first z, and the exponent bounds of p = z.
__global__ void __launch_bounds__(kRedThreads) k_first_scalars(PcgScalars* s, Partials bb, Partials rz) {
  const int k = blockIdx.x;
  const double b2 = warp_sum_partials(bb, k), z0 = warp_sum_partials(rz, k);
  int ex = kExpNone;
  if (rz.ex)
    for (int g = threadIdx.x; g < rz.n; g += kRedThreads) ex = max(ex, rz.ex[k * rz.pitch + g]);
  ex = block_max(ex);
  if (threadIdx.x != 0) return;
  const bool finite = isfinite(b2) && isfinite(z0);
  if (!finite) atomicOr(&s->flags, kErrNonFinite);
  s->bnorm2[k] = s->rr[k] = b2;
  s->rz[0][k] = z0;
  s->fz[k] = s->fp[0][k] = ex;
  s->fp[1][k] = kExpNone;
  s->conv[k] = !finite || b2 == 0.0;
  if (!s->conv[k]) atomicAdd(&s->running, 1);
}
__global__ void k_first_running(PcgScalars* s) { s->all_conv = s->running == 0; }

// The last iteration's convergence tests, where no direction update follows.
__global__ void __launch_bounds__(32) k_last_scalars(PcgScalars* s, Partials rrp, double tol2) {
  if (s->all_conv) return;
  const double rr = warp_sum_partials(rrp, blockIdx.x);
  if (threadIdx.x == 0) test_convergence(s, blockIdx.x, rr, tol2, true);
}

// x += alpha p, r -= alpha Ap with alpha from the partial sums of p . Ap, and
// partial sums of ||r||^2; block (g, k) its chunk of right-hand side k.
__global__ void __launch_bounds__(kRedThreads) k_update_xr(double* __restrict__ x, double* __restrict__ r,
                                                           const double* __restrict__ p, const double* __restrict__ Ap,
                                                           int64_t len, PcgScalars* s, Partials pap, Partials rrp,
                                                           int parity) {
  if (s->all_conv) return;
  const int k = blockIdx.y;
  const bool record = blockIdx.x == 0 && threadIdx.x == 0;
  __shared__ double s_alpha;
  if (threadIdx.x < 32) {
    const double sum = warp_sum_partials(pap, k);
    if (threadIdx.x == 0) s_alpha = take_alpha(s, k, sum, parity, record);
  }
  if (record) s->fp[parity ^ 1][k] = kExpNone;  // k_pcg_p gathers there
  __syncthreads();
  const double al = s_alpha;
  const int64_t o = (int64_t)k * len;
  int64_t i0, i1;
  chunk_of(len, i0, i1);
  double v = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    double rk = r[o + i];
    if (al != 0.0) {
      x[o + i] += al * p[o + i];
      rk -= al * Ap[o + i];
      r[o + i] = rk;
    }
    v += rk * rk;
  }
  v = block_sum(v);
  if (threadIdx.x == 0) rrp.sum[k * rrp.pitch + blockIdx.x] = v;
}

// The first split of p (p = z, |p| < 2^fz): fsplit = fz.
__global__ void __launch_bounds__(kRedThreads) k_split_p(const double* __restrict__ p, float2* __restrict__ ps,
                                                         const int32_t* __restrict__ kk, int64_t len, int nrhs,
                                                         PcgScalars* s) {
  const int k = blockIdx.y;
  const int F = s->fz[k] == kExpNone ? 0 : s->fz[k];
  if (blockIdx.x == 0 && threadIdx.x == 0) s->fsplit[k] = F;
  const int64_t o = (int64_t)k * len;
  int64_t i0, i1;
  chunk_of(len, i0, i1);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const uint32_t node = (uint32_t)i / 3u;
    ps[((int64_t)node * nrhs + k) * 3 + ((uint32_t)i - 3u * node)] = ff_split_bits(p[o + i], kk[node] - F);
  }
}

}  // namespace gs

using namespace gs;

extern "C" int gs_pcg_solve(gs_ctx ctx, gs_mat mat, gs_mas mas, const double* b, int32_t nrhs, double tol,
                            int32_t max_iter, int32_t variant, double* x, int32_t* iters, double* rel_res) {
  GS_CHECK(ctx && mat && mas && b && x, GS_ERR_INVALID, "gs_pcg_solve: null argument");
  GS_CHECK(nrhs >= 1 && nrhs <= kMaxRhs, GS_ERR_INVALID, "gs_pcg_solve: nrhs %d (1..%d)", nrhs, kMaxRhs);
  GS_CHECK(mas->n == mat->n, GS_ERR_INVALID, "gs_pcg_solve: preconditioner built for another size");
  GS_CHECK(tol >= 0.0 && max_iter >= 0, GS_ERR_INVALID, "gs_pcg_solve: tol %g max_iter %d", tol, max_iter);
  GS_CHECK(variant == GS_SPMV_SRBK || variant == GS_SPMV_ROW || variant == GS_SPMV_ROW_FF, GS_ERR_INVALID,
           "gs_pcg_solve: variant %d", variant);
  GS_CHECK(b != x, GS_ERR_INVALID, "gs_pcg_solve: b and x alias");
  GS_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  const int64_t len = 3LL * mat->n;
  const size_t vbytes = (size_t)nrhs * len * sizeof(double);
  const bool ff = variant == GS_SPMV_ROW_FF;
  double* vec = nullptr;
  GS_TRY(ctx->scratch_buf(kSlotPcgVectors, (ff ? 5 : 4) * vbytes, (void**)&vec));
  double *r = vec, *z = r + nrhs * len, *p = z + nrhs * len, *Ap = p + nrhs * len;
  float2* ps = (float2*)(Ap + nrhs * len);  // float-float operand (same size as a vector)
  // beyond kSmallWork the separate passes are faster: x, r streamed (55 us at
  // 64^3, 8 RHS), restricted (22), r . z streamed (22)
  const bool fused_mas = mas_dot_usable(ctx, mas, nrhs) && (int64_t)mat->n * nrhs <= kSmallWork;
  // scalars; partial sums of p . Ap, ||r||^2, r . z (per domain where the MAS
  // product takes it) and r . z folded
  const int rz_pitch = std::max(kMaxRedBlocks, fused_mas ? mas->n_domains[0] : 0);
  const size_t rows = (size_t)nrhs * (3 * kMaxRedBlocks + rz_pitch), erows = (size_t)nrhs * (kMaxRedBlocks + rz_pitch);
  char* sbuf = nullptr;
  GS_TRY(ctx->scratch_buf(kSlotPcgScalars, sizeof(PcgScalars) + 256 + rows * 8 + erows * 4, (void**)&sbuf));
  PcgScalars* s = (PcgScalars*)sbuf;
  double* sums = (double*)(sbuf + ((sizeof(PcgScalars) + 255) / 256) * 256);
  int* exps = (int*)(sums + rows);
  Partials pap, rrp, fold, rzp;
  pap.sum = sums, pap.pitch = kMaxRedBlocks;
  rrp.sum = sums + (size_t)nrhs * kMaxRedBlocks, rrp.pitch = kMaxRedBlocks;
  fold.sum = sums + 2 * (size_t)nrhs * kMaxRedBlocks, fold.ex = exps, fold.pitch = kMaxRedBlocks;
  rzp.sum = sums + 3 * (size_t)nrhs * kMaxRedBlocks, rzp.ex = exps + (size_t)nrhs * kMaxRedBlocks, rzp.pitch = rz_pitch;
  double *rl, *zl;
  GS_TRY(mas_level_vectors(ctx, mas, nrhs, &rl, &zl));
  GS_CUDA(cudaMemsetAsync(s, 0, sizeof(PcgScalars), st));
  // the sliced copy, built once per matrix, last of all: it is optional (without one the
  // product is a pass of its own) and must not take the room of what is not
  bool fused_spmv = nrhs <= 8 && variant != GS_SPMV_SRBK;
  if (fused_spmv) {
    GS_TRY(ensure_sliced(ctx, mat, ff));
    fused_spmv = ff ? mat->sl_ff != nullptr : mat->sl_f64 != nullptr;
  }
  if (!fused_spmv) {
    if (variant != GS_SPMV_SRBK) GS_TRY(ensure_row_order(ctx, mat));
    if (ff) GS_TRY(ensure_ff(ctx, mat));
  }

  const double tol2 = tol * tol;
  const dim3 vg(red_blocks(len, nrhs, ctx->sm_count), nrhs);
  rrp.n = rzp.n = vg.x;
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_init<<<vg, kRedThreads, 0, st>>>(b, x, r, len, rrp); }
  GS_TRY(mas_apply_launch(ctx, mas, r, z, nrhs, rl, zl));
  {
    GS_PROF(ctx, GS_K_PCG_VECTOR);
    if (ff)
      k_dot<true, true><<<vg, kRedThreads, 0, st>>>(r, z, p, len, nullptr, rzp);
    else
      k_dot<true, false><<<vg, kRedThreads, 0, st>>>(r, z, p, len, nullptr, rzp);
  }
  Partials rz0 = rzp;
  if (!ff) rz0.ex = nullptr, ps = nullptr;
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_first_scalars<<<nrhs, kRedThreads, 0, st>>>(s, rrp, rz0); }
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_first_running<<<1, 1, 0, st>>>(s); }
  if (ff) { GS_PROF(ctx, GS_K_PCG_VECTOR); k_split_p<<<vg, kRedThreads, 0, st>>>(p, ps, mat->ff_k, len, nrhs, s); }
  const int64_t lstride = 3 * std::max<int64_t>(mas->vec_items, 1);
  const int poll = 4;
  int* h_conv = ctx->h_pinned + 64;
  for (int q = 0; q < 2; ++q)
    if (!ctx->poll_event[q]) GS_CUDA(cudaEventCreateWithFlags(&ctx->poll_event[q], cudaEventDisableTiming));
  for (int it = 0, polls = 0; it < max_iter; ++it) {
    const int parity = it & 1;
    if (fused_spmv) {
      GS_TRY(pcg_spmv_dot(ctx, mat, ps, p, Ap, nrhs, s, pap));
    } else {
      if (ff)
        GS_TRY(spmv_ff_split_launch(ctx, mat, ps, s->fsplit, Ap, nrhs, &s->all_conv));
      else
        GS_TRY(spmv_launch_skip(ctx, mat, p, Ap, nrhs, variant, &s->all_conv));
      GS_PROF(ctx, GS_K_PCG_VECTOR);
      pap.n = vg.x;
      k_dot<false, false><<<vg, kRedThreads, 0, st>>>(p, Ap, nullptr, len, &s->all_conv, pap);
    }
    if (fused_mas) {
      GS_TRY(pcg_update_xr(ctx, mas, x, r, p, Ap, nrhs, rl, lstride, s, pap, rrp, parity));
    } else {
      GS_PROF(ctx, GS_K_PCG_VECTOR);
      k_update_xr<<<vg, kRedThreads, 0, st>>>(x, r, p, Ap, len, s, pap, rrp, parity);
    }
    if (it + 1 == max_iter) {
      GS_PROF(ctx, GS_K_PCG_VECTOR);
      k_last_scalars<<<nrhs, 32, 0, st>>>(s, rrp, tol2);
      break;
    }
    if (fused_mas) {
      rzp.n = mas->n_domains[0];
      GS_TRY(mas_products(ctx, mas, r, z, nrhs, rl, zl, &s->all_conv, &rzp));
    } else {
      GS_TRY(mas_apply_launch_skip(ctx, mas, r, z, nrhs, rl, zl, &s->all_conv));
      GS_PROF(ctx, GS_K_PCG_VECTOR);
      if (ff)
        k_dot<false, true><<<vg, kRedThreads, 0, st>>>(r, z, nullptr, len, &s->all_conv, rzp);
      else
        k_dot<false, false><<<vg, kRedThreads, 0, st>>>(r, z, nullptr, len, &s->all_conv, rzp);
    }
    GS_TRY(pcg_update_p(ctx, mat, p, z, ps, nrhs, s, rrp, rzp, fold, tol2, parity));
    if ((it + 1) % poll == 0) {
      const int q = polls++ & 1;
      GS_CUDA(cudaMemcpyAsync(h_conv + q, &s->all_conv, 4, cudaMemcpyDeviceToHost, st));
      GS_CUDA(cudaEventRecord(ctx->poll_event[q], st));
      if (polls > 1) {
        GS_CUDA(cudaEventSynchronize(ctx->poll_event[q ^ 1]));
        if (h_conv[q ^ 1]) break;
      }
    }
  }
  GS_CUDA(cudaGetLastError());
  // (h_pinned holds 4 KiB; its first words are the polls' and take_flags')
  PcgScalars* hp = (PcgScalars*)(ctx->h_pinned + 256);
  static_assert(1024 + sizeof(PcgScalars) <= 4096, "pinned staging");
  GS_CUDA(cudaMemcpyAsync(hp, s, sizeof(PcgScalars), cudaMemcpyDeviceToHost, st));
  int flags = 0;
  GS_TRY(ctx->take_flags(&flags));  // synchronises
  const PcgScalars& hs = *hp;
  bool all = true;
  for (int k = 0; k < nrhs; ++k) {
    if (iters) iters[k] = hs.iters[k];
    if (rel_res) rel_res[k] = hs.bnorm2[k] > 0 ? std::sqrt(hs.rr[k] / hs.bnorm2[k]) : 0.0;
    all = all && hs.conv[k];
  }
  if (hs.flags) return status_from_flags(hs.flags);
  if (flags) return status_from_flags(flags);
  if (!all) {
    set_error("gs_pcg_solve: not converged in %d iterations", max_iter);
    return GS_ERR_MAXITER;
  }
  return GS_OK;
}
