// M^-1 = W^T W of every domain of every level from the inverse Cholesky factors
// W that mas_invert.cu leaves in the matrices' place, one CTA per domain, in FP64
// accuracy on the F16 tensor cores; and the digit bytes of the result.
//
// W^T W is a third of the inversion's FP64 instructions, which are all that
// bounds it.  Column i of W gets an exponent c_i with |W_ki| < 2^(c_i - 1);
// X_ki = rint(W_ki 2^(56 - c_i)) is cut into 7 balanced base-256 digits, F16
// (exact), and one K-major copy of the digit matrices X^T serves as both operands:
//   G_s = sum_{p + q = s} (X^p)^T X^q,  s = 2 .. 9,
// products of digits <= 2^14, 96 terms, <= 7 pairs: exact in FP32.  M^-1_ij =
// 2^(c_i + c_j - 72) sum_s G_s 256^(9-s), combined in 64-bit integers and rounded
// once.  The roundings of X, 96 of half a unit on either operand against magnitudes
// up to 2^55, come to 96 2^-57 of 2^(c_i + c_j) at most, the dropped terms to 2^-57;
// 2^(2 c_i) <= 16 max W_ki^2 <= 16 M^-1_ii, so the bound is 96 2^-53 sqrt(M^-1_ii
// M^-1_jj), that of the sum in FP64 (2^-57 16 beyond it).
//
// The groups 2 .. 6 fill the tensor memory (5 x 96 of 512 columns); 2 .. 5 are read
// as the result's high part while 6 is formed, then 7 .. 9 take their place.  W is
// lower triangular: K step ks has columns j < 16 (ks + 1) only.  Reading the A
// operand from shared memory costs an MMA 32 clocks however many columns it has,
// so all 96 columns at once (a third of them at a time: 408 MMAs of 50 clocks
// instead of 204 of 46).  The digits take 129 KB of shared memory: one CTA of 1024
// threads per SM.  What bounds it is integer work on those threads (the digits, the
// rounding of the results, the digit bytes) more than the MMAs.  Build of a 64^3
// body, 8,456 domains: 10.25 ms with the product in FP64, 9.10 with this (9.26 with
// 512 threads, 9.54 column by column); the inversions of a 32^3 body 1.10 ms before,
// 0.78 + 0.20 now.
#include <algorithm>

#include "common.cuh"
#include "fp64split.cuh"
#include "primitives.cuh"
#include "square.cuh"
#include "umma.cuh"

namespace gs {
namespace square {

constexpr int kThreads = 1024;
constexpr int kWarps = kThreads / 32;
constexpr int kDigits = 7;
constexpr int kM = 128;
constexpr int kNone = -100000;  // exponent of an all-zero row or column

__device__ __forceinline__ int tri(int i, int j) { return i * (i + 1) / 2 + j; }

// rows LD .. 127 of the A operand are read (and not used) past the last digit
__host__ __device__ constexpr uint32_t digits_bytes(int ld) { return (uint32_t)(kDigits * ld * ld * 2 + (kM - ld) * 16); }
__host__ __device__ constexpr size_t smem_bytes(int ld) { return 128 + digits_bytes(ld) + (size_t)ld * (ld + 1) * 8; }

template <int LD>
__global__ void __launch_bounds__(kThreads, 1) k_square_factors(Jobs jb, const int32_t* __restrict__ remap0,
                                                                int* __restrict__ flags) {
  using namespace umma;
  constexpr int ld = LD, N = LD / 3;
  constexpr int kCols = LD == 96 ? 512 : 256, kSteps = LD / 16, kRowWarps = (LD + 31) / 32;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sD = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  double* sW = (double*)(sD + digits_bytes(LD));  // packed lower triangle of W, then of the result's high parts and it
  long long* sL = (long long*)(sW + LD * (LD + 1) / 2);  // its low parts
  __shared__ int s_col[LD], s_exp[LD], s_lane[32], s_pos[32], s_k;
  __shared__ uint64_t bar[3];
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  int l = 0;
  while (l + 1 < jb.L && (int)blockIdx.x >= jb.first[l + 1]) ++l;
  const int64_t d = blockIdx.x - jb.first[l];
  double* M = jb.mat[l] + d * ld * ld;
  if (tid < 32) {
    const bool real = tid < N && (l == 0 ? remap0[d * N + tid] >= 0 : d * N + tid < jb.n_items[l]);
    const uint32_t rm = __ballot_sync(kFull, real);
    const int pos = __popc(rm & ((1u << tid) - 1u));
    if (real) s_lane[pos] = tid;
    s_pos[tid] = real ? pos : -1;
    if (tid == 0) s_k = __popc(rm);
  }
  if (tid == 32) {
    for (int c = 0; c < 3; ++c) mbar_init(&bar[c], 1);
    fence_mbar_init();
  }
  if (wid == 2) {
    tmem_alloc(&tslot, kCols);
    tmem_relinquish();
  }
  for (int i = tid; i < LD; i += kThreads) s_exp[i] = kNone;
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = tslot;
  const int n3 = 3 * s_k, np = (n3 + 7) / 8 * 8;
  for (int i = tid; i < np * (np + 1) / 2; i += kThreads) sW[i] = M[i];
  __syncthreads();
#pragma unroll
  for (int u = 0; u < (LD + kWarps - 1) / kWarps; ++u) {  // column exponents
    const int i = wid + kWarps * u;
    if (i >= LD) break;  // whole warp
    int top = 0;
#pragma unroll
    for (int v = 0; v < (LD + 31) / 32; ++v) {
      const int k = lane + 32 * v;
      if (k >= i && k < np) top = max(top, __double2hiint(sW[tri(k, i)]) & 0x7FFFFFFF);
    }
    top = __reduce_max_sync(kFull, top);
    if (lane == 0) s_col[i] = top >> 20 ? (top >> 20) - 1021 : kNone;
  }
  __syncthreads();
  // digit matrices, element (i, k) = digit of W_ki at (k/8) (16 LD) + (i/8) 128 +
  // (i%8) 16 + (k%8) 2: a warp per 8 x 8 tile, a lane two neighbouring k of one i
  constexpr int G = LD / 8;
  for (int t = wid; t < G * G; t += kWarps) {
    const int Ib = t % G, Kb = t / G, i = 8 * Ib + (lane >> 2), k = 8 * Kb + 2 * (lane & 3);
    uint32_t* o = (uint32_t*)(sD + Kb * (16 * LD) + Ib * 128) + lane;
    if (Kb < Ib || 8 * Kb >= np) {  // whole warp
#pragma unroll
      for (int p = 0; p < kDigits; ++p) o[p * (LD * LD / 2)] = 0;
      continue;
    }
    unsigned long long z[2] = {kBias256, kBias256};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (k + h >= i) z[h] = (unsigned long long)scaled_rint(sW[tri(k + h, i)], s_col[i]) + kBias256;
    }
    // 1024 + 128 + digit as F16, less 1152; the leading digit may be 128
    const uint32_t l0 = (uint32_t)z[0], l1 = (uint32_t)z[1], h0 = (uint32_t)(z[0] >> 32), h1 = (uint32_t)(z[1] >> 32);
    const uint32_t off = 0x64806480u;
#pragma unroll
    for (int p = 0; p < kDigits; ++p) {
      const int q = 6 - p;  // byte
      const uint32_t pair = q < 4 ? __byte_perm(l0, l1, q | (q + 4) << 4) : __byte_perm(h0, h1, (q - 4) | q << 4);
      const uint32_t w = p ? __byte_perm(pair, 0x64646464u, 0x4140) : (0x6400u + (h0 >> 16)) | (0x6400u + (h1 >> 16)) << 16;
      const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&w), *reinterpret_cast<const __half2*>(&off));
      o[p * (LD * LD / 2)] = *reinterpret_cast<const uint32_t*>(&v);
    }
  }
  fence_proxy_async();
  __syncthreads();  // W is in the digits: its place takes the result

  auto place = [](int s) { return (uint32_t)(s < 5 ? s : s - 5) * LD; };  // columns of group s + 2
  auto issue = [&](int s0, int s1, uint64_t* done) {                     // one thread: groups s0 + 2 .. s1 + 2
    const uint64_t d0 = smem_desc(smem_u32(sD), 16 * LD, 128);
#pragma unroll 1
    for (int s = s0; s <= s1; ++s)
#pragma unroll 1
      for (int p = max(0, s - 6); p <= min(s, 6); ++p) {
        const uint64_t da = d0 + ((uint32_t)p * (LD * LD * 2) >> 4), db = d0 + ((uint32_t)(s - p) * (LD * LD * 2) >> 4);
#pragma unroll
        for (int ks = kSteps - 1; ks >= 0; --ks)  // the last step first: it has all the columns
          mma_f16(tmem + place(s), da + ks * (32u * LD >> 4), db + ks * (32u * LD >> 4), idesc_f16_f32(kM, 16 * (ks + 1)),
                  p == max(0, s - 6) && ks == kSteps - 1 ? 0u : 1u);
      }
    mma_commit(done);
  };
  const int q4 = wid & 3, part = wid >> 2, i = q4 * 32 + lane;
  const bool rows = q4 < kRowWarps;  // whole warp
  bool ok = true;
  // this thread's row, every eighth group of four columns up to the diagonal: the
  // weighted sum of four groups
  auto read = [&](bool low) {
    fence_after_sync();
#pragma unroll 1
    for (int j0 = 4 * part; j0 < LD && j0 <= q4 * 32 + 31; j0 += kWarps) {  // whole warp
      float g[16];
      uint32_t at[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) at[s] = tmem + ((uint32_t)(q4 * 32) << 16) + place(s + (low ? 4 : 0)) + j0;
      tmem_ld_32x32b_4x4(at, g);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int j = j0 + u;
        if (i >= np || j > i) continue;
        long long sum = __float2int_rn(g[12 + u]);
#pragma unroll
        for (int s = 0; s < 3; ++s) sum += (long long)__float2int_rn(g[4 * s + u]) * (1 << (24 - 8 * s));
        if (low)
          sL[tri(i, j)] = sum;
        else
          sW[tri(i, j)] = __longlong_as_double(sum);
      }
    }
  };
  if (tid == 96) {  // warp 3 owns no rows
    issue(0, 3, &bar[0]);
    issue(4, 4, &bar[1]);
  }
  __syncwarp();
  if (rows) {
    ok = __all_sync(kFull, mbar_wait(&bar[0], 0));
    if (ok) read(false);
  }
  fence_before_sync();
  __syncthreads();
  if (tid == 96) {
    fence_after_sync();
    issue(5, 7, &bar[2]);
  }
  __syncwarp();
  if (rows) {
    ok = ok && __all_sync(kFull, mbar_wait(&bar[1], 0) && mbar_wait(&bar[2], 0));
    if (ok) read(true);
    if (!ok && lane == 0) atomicOr(flags, kErrTimeout);
  }
  if (wid == 3) {  // every MMA ends before the CTA leaves
    const bool end = mbar_wait(&bar[2], 0) && mbar_wait(&bar[1], 0);
    if (!end && lane == 0) atomicOr(flags, kErrTimeout);
  }
  fence_before_sync();
  __syncthreads();
  if (wid == 2) {
    fence_after_sync();
    tmem_dealloc(tmem, kCols);
  }
  // the two parts as a double, a warp per row (the rows' own warps are three of
  // every four, and the last of them has most of the triangle)
  for (int r = wid; r < np; r += kWarps)
    for (int j = lane; j <= r; j += 32) {
      const int c = s_col[r] > kNone && s_col[j] > kNone ? s_col[r] + s_col[j] - 72 : kNone;
      double* m = sW + tri(r, j);
      *m = c > kNone ? combine_to_double(__double_as_longlong(*m), sL[tri(r, j)], 32, c) : 0.0;
    }
  __syncthreads();

  // the matrix whole, zeros in the padding (a warp per row), and the row's
  // exponent a: |M_ij| < 2^(a - 1), and |M_ij| 2^(56 - a) so far below 2^55 that its
  // leading balanced digit is at most 127 (the bytes hold -128 .. 127): rows whose
  // largest magnitude has a mantissa of 0xFDFDF.. or more, 1.992 of 2, take one more
  uint8_t* dig = jb.dig[l];
  for (int gi = wid; gi < LD; gi += kWarps) {
    const int ni = s_pos[gi / 3], a = 3 * ni + gi % 3;
    int top = 0;  // sign-free upper words order like the magnitudes
    for (int gj = lane; gj < LD; gj += 32) {
      const int nj = s_pos[gj / 3], b = 3 * nj + gj % 3;
      const double v = ni >= 0 && nj >= 0 ? sW[b <= a ? tri(a, b) : tri(b, a)] : 0.0;
      M[gi * LD + gj] = v;
      top = max(top, __double2hiint(v) & 0x7FFFFFFF);
    }
    top = __reduce_max_sync(kFull, top);
    if (lane == 0 && top >> 20) s_exp[gi] = (top >> 20) - 1021 + ((top & 0xFFFFF) >= 0xFDFDF);
  }
  if (!dig) return;
  __syncthreads();
  if (tid < LD) jb.dexp[l][d * LD + tid] = s_exp[tid];
  // digit matrices in the order their rows are loaded (mas_apply_f64tc.cu):
  // [k/16][i][k%16] bytes; a warp takes 8 rows by 16 columns, 128 contiguous
  // bytes per digit, a lane four neighbouring columns of a row
  uint8_t* out = dig + d * kDigits * (LD * LD);
  for (int t = wid; t < G * (LD / 16); t += kWarps) {
    const int gi = 8 * (t % G) + (lane >> 2), gk = 16 * (t / G) + 4 * (lane & 3);
    const int ni = s_pos[gi / 3], a = s_exp[gi];
    unsigned long long z[4];  // the digits + 128, one byte each
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int nk = s_pos[(gk + h) / 3];
      long long x = 0;
      if (ni >= 0 && nk >= 0 && a > kNone) {
        const int r = 3 * ni + gi % 3, k = 3 * nk + (gk + h) % 3;
        x = scaled_rint(sW[k <= r ? tri(r, k) : tri(k, r)], a);
      }
      z[h] = (unsigned long long)x + kBias256;
    }
    uint8_t* o = out + ((t / G) * LD + gi) * 16 + 4 * (lane & 3);
    uint32_t w[7];
    bytes_of_four(z, w);
#pragma unroll
    for (int p = 0; p < kDigits; ++p) *(uint32_t*)(o + p * (LD * LD)) = w[p];
  }
}

template <int LD>
static int launch(gs_ctx ctx, const Jobs& jb, const int32_t* remap0) {
  const size_t smem = smem_bytes(LD);
  GS_CUDA(cudaFuncSetAttribute(k_square_factors<LD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_square_factors<LD><<<jb.first[jb.L], kThreads, smem, ctx->stream>>>(jb, remap0, ctx->d_flags);
  GS_CUDA(cudaGetLastError());
  return GS_OK;
}

}  // namespace square

int square_factors_launch(gs_ctx ctx, const square::Jobs& jb, int N, const int32_t* remap0) {
  return N == 32 ? square::launch<96>(ctx, jb, remap0) : square::launch<48>(ctx, jb, remap0);
}

}  // namespace gs
