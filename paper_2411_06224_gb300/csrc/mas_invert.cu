// Domain inverses of the MAS preconditioner (Alg. 1 "invert unpadded parts"),
// one CTA per domain of every level.
//
// The real part of a domain matrix (3k x 3k, 3k <= 96) is factorised in
// shared memory (Cholesky, FP64) and the factor inverted, W = L^-1.  For domains
// of 16 and 32 nodes W is written over the matrix and mas_square.cu forms W^T W =
// M^-1 on the tensor cores; for other sizes W^T W is formed here.  Rows beyond 3k
// up to the next multiple of 8 hold the identity, so every step works on whole 8 x
// 8 tiles.
//
// What bounds it: FP64 arithmetic, (3k)^3 / 6 FMA per domain and product at 2 per
// clock and SM (4.0 ms for the two products and the 8,456 domains of a 64^3 body),
// where an instruction costs its 16 cycles however few lanes take part.  So the
// products run on tiles whose 32 lanes all work (lane (r, c) owns entries (r, c)
// and (r, c + 4)), with a few block barriers per 8 columns instead of three per
// column; square roots and reciprocals, 96 one-lane chains of a library division
// and square root before, are one chain of a few FMA per column.  Measured on the
// 1,060 domains of a 32^3 body: 0.78 ms (all three products 1.10, column by column
// and with a separate digit pass 1.72 + 0.09).
#include <algorithm>

#include "common.cuh"
#include "fp64split.cuh"
#include "primitives.cuh"
#include "square.cuh"

namespace gs {

int square_factors_launch(gs_ctx ctx, const square::Jobs& jb, int N, const int32_t* remap0);

namespace invert {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxRows = 96;  // 3 N, N <= 32

using square::Jobs;

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }

// v 2^k for a normal v whose scaled value stays normal.
__device__ __forceinline__ double scale_exp(double v, int k) {
  return __hiloint2double(__double2hiint(v) + k * (1 << 20), __double2loint(v));
}

// sqrt(d) and 1 / sqrt(d) of a positive d, each within a few units of the
// last place: d = m 4^k with m in [1, 4), a single-precision 1 / sqrt(m) as
// the start, one third-order Householder step y (1 + e/2 + 3/8 e^2) with
// e = 1 - m y^2, and one Newton correction of the root.  About ten FP64
// instructions in one chain; the library's square root and division take
// several times that.
__device__ __forceinline__ void sqrt_and_inverse(double d, double& root, double& inv) {
  const int ef = (__double2hiint(d) >> 20) & 0x7ff;
  if (ef == 0 || ef == 0x7ff) {  // subnormal or infinite
    root = sqrt(d);
    inv = 1.0 / root;
    return;
  }
  const int k = (ef - 1023) >> 1;
  const double m = scale_exp(d, -2 * k);
  const double y0 = f32_to_f64_bits(rsqrtf(f64_to_f32_bits(m)));
  const double t = m * y0;
  const double e = fma(-t, y0, 1.0);
  const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);
  double s = m * y;
  s = fma(fma(-s, s, m), 0.5 * y, s);
  root = scale_exp(s, k);
  inv = scale_exp(y, -k);
}

// kSquare: the inverses; else the factors W, packed by rows in the matrices' place.
template <bool kSquare>
__global__ void __launch_bounds__(kThreads, 4) k_invert_domains(Jobs jb, const int32_t* __restrict__ remap0,
                                                                int* __restrict__ flags, double* __restrict__ fac0) {
  extern __shared__ double sA[];  // lower triangle packed by rows: (i, j), j <= i, at i (i + 1) / 2 + j
  __shared__ double s_inv[kMaxRows];  // 1 / L_ii
  __shared__ int s_lane[32];          // compacted node -> lane of the domain
  __shared__ int s_k, s_bad;
  const int job = blockIdx.x;
  int l = 0;
  while (l + 1 < jb.L && job >= jb.first[l + 1]) ++l;
  const int64_t d = job - jb.first[l];
  const int N = jb.N, ld = 3 * N;
  double* M = jb.mat[l] + d * ld * ld;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int tr = lane >> 2, tc = lane & 3;  // this lane's row and first column in a tile
  if (tid < 32) {
    const bool real = tid < N && (l == 0 ? remap0[d * N + tid] >= 0 : d * N + tid < jb.n_items[l]);
    const uint32_t rm = __ballot_sync(kFull, real);
    const int pos = __popc(rm & ((1u << tid) - 1u));
    if (real) s_lane[pos] = tid;
    if (tid == 0) s_k = __popc(rm), s_bad = 0;
  }
  __syncthreads();
  const int n3 = 3 * s_k, nb = (n3 + 7) / 8, np = 8 * nb;
  for (int i = wid; i < np; i += kWarps) {
    const int gi = i < n3 ? 3 * s_lane[i / 3] + i % 3 : 0;
    for (int j = lane; j <= i; j += 32)
      sA[tri(i, j)] = i < n3 ? M[(int64_t)gi * ld + 3 * s_lane[j / 3] + j % 3] : (i == j ? 1.0 : 0.0);
  }
  if (tid < 8) sA[tri(np, tid)] = 0.0;  // read (and not used) past the last row's diagonal
  __syncthreads();

  // Cholesky by panels of 8 columns: A_IK -= sum_p L_Ip L_Kp^T over the
  // columns before the panel, the 8 x 8 diagonal block in one warp's
  // registers, then a thread per row below for the panel's triangular solve.
  for (int K = 0; K < nb; ++K) {
    if (K > 0) {
      for (int I = K + wid; I < nb; I += kWarps) {
        const int i = 8 * I + tr, j0 = 8 * K + tc, j1 = j0 + 4;
        const double *ri = sA + tri(i, 0), *r0 = sA + tri(j0, 0), *r1 = sA + tri(j1, 0);
        double a0 = ri[j0], a1 = ri[j1];
#pragma unroll 8
        for (int p = 0; p < 8 * K; ++p) {
          const double v = ri[p];
          a0 = fma(-v, r0[p], a0);
          a1 = fma(-v, r1[p], a1);
        }
        __syncwarp();  // an entry above the diagonal read a neighbour's
        if (j0 <= i) sA[tri(i, j0)] = a0;
        if (j1 <= i) sA[tri(i, j1)] = a1;
      }
      __syncthreads();
    }
    if (wid == 0) {
      const int r = lane & 7;
      double* row = sA + tri(8 * K + r, 8 * K);
      double a[8];
      bool bad = false;
#pragma unroll
      for (int c = 0; c < 8; ++c) a[c] = c <= r ? row[c] : 0.0;
      __syncwarp();
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        double dpp = __shfl_sync(kFull, a[c], c);
        if (!(dpp > 0.0)) bad = true, dpp = 1.0;
        double lpp, inv;
        sqrt_and_inverse(dpp, lpp, inv);
        a[c] = r == c ? lpp : a[c] * inv;
        if (lane == c) s_inv[8 * K + c] = inv;
#pragma unroll
        for (int q = c + 1; q < 8; ++q) a[q] = fma(-a[c], __shfl_sync(kFull, a[c], q), a[q]);
      }
      if (lane < 8) {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (c <= r) row[c] = a[c];
      }
      if (bad && lane == 0) s_bad = 1;
    }
    __syncthreads();
    if (s_bad) break;
    const int i = 8 * (K + 1) + tid;
    if (i < np) {
      double* row = sA + tri(i, 8 * K);
      double x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = row[c];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const double* lc = sA + tri(8 * K + c, 8 * K);
        double v = x[c];
#pragma unroll
        for (int q = 0; q < c; ++q) v = fma(-x[q], lc[q], v);
        x[c] = v * s_inv[8 * K + c];
        row[c] = x[c];
      }
    }
    __syncthreads();
  }
  if (s_bad) {
    if (tid == 0) atomicOr(flags, kErrNotSPD);
    return;
  }

  // W = L^-1 in place: the diagonal blocks first (a thread per column), then
  // row block by row block W_IJ = -W_II sum_{Q=J..I-1} L_IQ W_QJ.
  if (tid < np) {
    const int b8 = tid & ~7, c = tid & 7;
    double w[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const double* lr = sA + tri(b8 + r, b8);
      double s = 0.0;
#pragma unroll
      for (int q = 0; q < r; ++q) s = fma(lr[q], w[q], s);
      const double ir = s_inv[b8 + r];
      w[r] = r < c ? 0.0 : (r == c ? ir : -s * ir);
    }
    const int left = np - (tid & ~31);  // active lanes of this warp (a multiple of 8)
    __syncwarp(left >= 32 ? kFull : (1u << left) - 1u);
#pragma unroll
    for (int r = 0; r < 8; ++r)
      if (r >= c) sA[tri(b8 + r, b8 + c)] = w[r];
  }
  __syncthreads();
  for (int I = 1; I < nb; ++I) {
    const int i = 8 * I + tr;
    const double* ri = sA + tri(i, 0);
    double t[2][2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int J = wid + kWarps * u;
      if (J >= I) break;  // whole warp
      const int j0 = 8 * J + tc, j1 = j0 + 4;
      double s0 = 0.0, s1 = 0.0;
      const double* rq = sA + tri(8 * J, 0);
#pragma unroll
      for (int q = 8 * J, z = 0; z < 8; ++z, ++q) {  // W_JJ is lower triangular
        const double v = ri[q];
        s0 = fma(v, q >= j0 ? rq[j0] : 0.0, s0);
        s1 = fma(v, q >= j1 ? rq[j1] : 0.0, s1);
        rq += q + 1;
      }
#pragma unroll 8
      for (int q = 8 * (J + 1); q < 8 * I; ++q) {
        const double v = ri[q];
        s0 = fma(v, rq[j0], s0);
        s1 = fma(v, rq[j1], s1);
        rq += q + 1;
      }
      double t0 = 0.0, t1 = 0.0;
      const double* wr = ri + 8 * I;  // row tr of W_II
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const double v = s <= tr ? wr[s] : 0.0;
        t0 = fma(-v, __shfl_sync(kFull, s0, 4 * s + tc), t0);
        t1 = fma(-v, __shfl_sync(kFull, s1, 4 * s + tc), t1);
      }
      t[u][0] = t0, t[u][1] = t1;
    }
    __syncthreads();  // L_IQ and W_II read by every warp
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int J = wid + kWarps * u;
      if (J >= I) break;
      sA[tri(i, 8 * J + tc)] = t[u][0];
      sA[tri(i, 8 * J + tc + 4)] = t[u][1];
    }
    __syncthreads();
  }
  // level 0, low-precision form: keep the factor W (M^-1 = W^T W)
  if (fac0 && l == 0) {
    double* F = fac0 + d * ld * ld;
    for (int i = wid; i < n3; i += kWarps) {
      const int gi = 3 * s_lane[i / 3] + i % 3;
      for (int j = lane; j <= i; j += 32) F[(int64_t)gi * ld + 3 * s_lane[j / 3] + j % 3] = sA[tri(i, j)];
    }
  }

  if (!kSquare) {
    for (int i = tid; i < np * (np + 1) / 2; i += kThreads) M[i] = sA[i];
    return;
  }

  // Inverse = W^T W, lower triangle, in place.  Tile (I, J) reads rows
  // 8 I .. of W, so the row blocks 0..7 can be overwritten before the tiles of
  // the last row blocks are formed; each warp holds its tiles of one half in
  // registers until every warp has read.
  const int half = min(nb, 8);
#pragma unroll 1
  for (int part = 0; part < 2; ++part) {
    const int t0 = part ? half * (half + 1) / 2 : 0, t1 = part ? nb * (nb + 1) / 2 : half * (half + 1) / 2;
    double acc[6][2];
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const int t = t0 + wid + kWarps * u;
      if (t >= t1) break;  // whole warp
      int I = 0;
      while ((I + 1) * (I + 2) / 2 <= t) ++I;
      const int J = t - I * (I + 1) / 2;
      const int i = 8 * I + tr, j0 = 8 * J + tc, j1 = j0 + 4;
      double s0 = 0.0, s1 = 0.0;
      const double* rq = sA + tri(8 * I, 0);
#pragma unroll
      for (int q = 8 * I, z = 0; z < 8; ++z, ++q) {
        const double v = q >= i ? rq[i] : 0.0;
        s0 = fma(v, q >= j0 ? rq[j0] : 0.0, s0);
        s1 = fma(v, q >= j1 ? rq[j1] : 0.0, s1);
        rq += q + 1;
      }
#pragma unroll 8
      for (int q = 8 * (I + 1); q < np; ++q) {
        const double v = rq[i];
        s0 = fma(v, rq[j0], s0);
        s1 = fma(v, rq[j1], s1);
        rq += q + 1;
      }
      acc[u][0] = s0, acc[u][1] = s1;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 6; ++u) {
      const int t = t0 + wid + kWarps * u;
      if (t >= t1) break;
      int I = 0;
      while ((I + 1) * (I + 2) / 2 <= t) ++I;
      const int J = t - I * (I + 1) / 2;
      const int i = 8 * I + tr, j0 = 8 * J + tc, j1 = j0 + 4;
      if (j0 <= i) sA[tri(i, j0)] = acc[u][0];
      if (j1 <= i) sA[tri(i, j1)] = acc[u][1];
    }
    // the second half reads rows 64.. only, the first half wrote the rows before
  }
  __syncthreads();

  // both triangles over the real part of the matrix (a warp per row)
  for (int i = wid; i < n3; i += kWarps) {
    const int gi = 3 * s_lane[i / 3] + i % 3;
    for (int j = lane; j < n3; j += 32) M[(int64_t)gi * ld + 3 * s_lane[j / 3] + j % 3] = sA[j <= i ? tri(i, j) : tri(j, i)];
  }
}

}  // namespace invert

// Inverts every level matrix of `mas` in place (mas->inv64); fac0, if not
// null, receives the level-0 factors W.  Where digit storage was made
// (mas->dig64), the digit matrices and row exponents are written as well.
int invert_domains_launch(gs_ctx ctx, gs_mas mas, double* fac0) {
  invert::Jobs jb{};
  jb.L = mas->L;
  jb.N = mas->N;
  for (int l = 0; l < mas->L; ++l) {
    jb.mat[l] = mas->inv64[l];
    jb.dig[l] = mas->dig64.empty() ? nullptr : (uint8_t*)mas->dig64[l];
    jb.dexp[l] = mas->dig64_exp.empty() ? nullptr : mas->dig64_exp[l];
    jb.n_items[l] = mas->n_items[l];
    jb.first[l + 1] = jb.first[l] + mas->n_domains[l];
  }
  const int np = (3 * mas->N + 7) / 8 * 8;
  const size_t smem = ((size_t)np * (np + 1) / 2 + 8) * sizeof(double);
  GS_PROF(ctx, GS_K_MAS_INVERT);
  const bool factors = mas->N == 16 || mas->N == 32;  // the tensor cores square them
  (factors ? invert::k_invert_domains<false> : invert::k_invert_domains<true>)<<<jb.first[mas->L], invert::kThreads,
                                                                                smem, ctx->stream>>>(
      jb, mas->remap0, ctx->d_flags, fac0);
  GS_CUDA(cudaGetLastError());
  if (factors) GS_TRY(square_factors_launch(ctx, jb, mas->N, mas->remap0));
  return GS_OK;
}

}  // namespace gs
