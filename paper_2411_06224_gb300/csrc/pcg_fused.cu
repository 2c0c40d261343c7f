// The kernels of one PCG iteration (pcg.cu):
//   k_pcg_spmv   Ap = A p (row or float-float product over the sliced matrix),
//                partial sums of p . Ap
//   k_pcg_xr     alpha from those; x += alpha p, r -= alpha Ap, partial sums of
//                ||r||^2, and the level-1 sums of r, a warp per level-0 domain
//   (the MAS products, the level-0 one with partial sums of r . z)
//   k_pcg_p      the convergence test and beta from the partial sums; p = z +
//                beta p (and the float-float operand of the next product)
//
// What bounds them: on small systems the chain of launches and reductions (ten
// launches of 6 to 8 us each per iteration before, five now), on large ones
// the vectors' bytes and the FP64 pipe.  A reduction has no tail: a kernel
// writes its partial sums (block b's covers a fixed share of the rows or
// domains), and every block of the kernel that needs the scalar adds them in
// the same fixed order, so all see the same bits.  What a kernel reads that is
// older than the kernel just before it is loaded before that one has ended.
// Per iteration, before and now: 16^3, 4 RHS 110 / 42 us; 40^3, 4 RHS, FP32
// preconditioner 205 / 119; 45^3, 1 RHS 197 / 121; 64^3, 8 RHS 655 / 547.
#include <algorithm>

#include "common.cuh"
#include "ff_product.cuh"
#include "pcg_state.cuh"

namespace gs {

constexpr int kT = 256;
constexpr int kWarps = kT / 32;

// ---------------------------------------------------------------- Ap = A p, p . Ap
struct Sliced {  // the sliced matrix (sliced.cu)
  const int32_t *row_order, *ptr, *len, *col;
  const float2* ff;
  const double* f64;
  int32_t n;
};

// One row by kBL * kRL lanes: kRL groups take kR right-hand sides each, the kBL
// lanes of a group share the row's entries and merge in a fixed order.  kFF:
// float-float (spmv_ff.cu), xs the split operand; else FP64, x the operand.  A lane
// that sums a whole row gathers twice the small parts that each of two lanes
// would, with as much more rounding, so its pairs are settled every kSettle entries
// (where 2 or 4 lanes share it, not: the chain is short, and the loop in pieces cost
// 3 % at 40^3, 1 RHS).
// 64^3, 8 RHS, 24 iterations: error 9.4e-14, 13.13 ms (1.7e-13 and 13.12 with three
// roundings a term at the size of L and never settled; 1.16e-13 with two lanes to a
// row; settling every fourth entry 5.8e-14 and 13.4).  An
// entry's column is loaded one entry ahead, so that its operand's gather leaves
// with the entry's own values.
constexpr int kSettle = 16;
template <bool kFF, int kBL, int kRL, int kR, int kThreads, int kMin>
__global__ void __launch_bounds__(kThreads, kMin) k_pcg_spmv(Sliced A, const int32_t* __restrict__ kk,
                                                             const float2* xs, const double* p,
                                                             double* __restrict__ Ap, int64_t stride, int nrhs,
                                                             const PcgScalars* s, Partials pap) {
  constexpr int G = kBL * kRL;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane % G;
  const int bl = sub % kBL, r0 = sub / kBL * kR;
  const int nh = min(kR, nrhs - r0);  // may be <= 0
  // an FP64 row's sums end up in two of its lanes, half of the right-hand sides each:
  // half the additions and products of p . Ap (53^3, 7 RHS: 12.55 -> 12.2 ms)
  constexpr bool kHalves = !kFF && kBL > 1;
  constexpr int kH = kHalves ? (kR + 1) / 2 : kR;
  const bool up = kHalves && (bl & 1), holds = bl < (kHalves ? 2 : 1);
  const int q0 = up ? kH : 0;
  const bool vec = kR % 2 == 0 && (nrhs & 1) == 0;
  double dot[kH];
#pragma unroll
  for (int q = 0; q < kH; ++q) dot[q] = 0.0;
  const int64_t chunks = ((int64_t)A.n * G + kThreads - 1) / kThreads;
  // blocks take one chunk of every gridDim.x, another place of it each time
  // (rows are ordered by length within windows: the same place would always
  // meet the same lengths)
  const int64_t rounds = (chunks + gridDim.x - 1) / gridDim.x;
  int32_t len, row, next;
  int64_t base;  // entry 0 of the row
  auto open_row = [&](int64_t i) {
    const int64_t c = i * gridDim.x + (blockIdx.x + i * 37) % gridDim.x;
    const int64_t slot = c * (kThreads / G) + threadIdx.x / G;
    const bool in = c < chunks && slot < A.n && nh > 0;
    len = in ? A.len[slot] : 0;
    base = in ? (int64_t)A.ptr[slot >> 5] * 32 + (slot & 31) : 0;
    row = in ? A.row_order[slot] : -1;
    next = bl < len ? A.col[base + 32 * bl] : 0;
  };
  open_row(0);  // the matrix is older than the kernel before
  wait_for_previous_kernel();
  if (s->all_conv) return;
  for (int64_t i = 0; i < rounds; ++i) {
    if (i > 0) open_row(i);
    const bool in = row >= 0;
    const int32_t lane_slot = (int32_t)(base & 31);
    double y[kR * 3];
    if (kFF) {
      FFSum<kR * 3> acc;
      acc.clear();
      const float2* v = A.ff + (base - lane_slot) * 9 + lane_slot;
      for (int32_t e = bl; e < len;) {
        const int32_t end = kBL == 1 ? min(len, e + kSettle) : len;
        for (; e < end; e += kBL) {
          const int32_t col = next;
          if (e + kBL < len) next = A.col[base + 32 * (int64_t)(e + kBL)];
          float2 H[9];
#pragma unroll
          for (int q = 0; q < 9; ++q) H[q] = v[(int64_t)e * 288 + 32 * q];
          ff_block_product<kR>(H, xs + ((int64_t)col * nrhs + r0) * 3, nh, vec, acc);
        }
        if (kBL == 1) acc.settle();
      }
      acc.template merge<kBL>();
      if (in && bl == 0) {
        const int kr = kk[row] + 2 * kk[A.n];  // k_row + K
#pragma unroll
        for (int q = 0; q < kR; ++q) {
          const int f = q < nh ? s->fsplit[r0 + q] : kExpNone;
#pragma unroll
          for (int j = 0; j < 3; ++j) y[3 * q + j] = f == kExpNone ? 0.0 : acc.value(3 * q + j, kr + f);
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < kR * 3; ++q) y[q] = 0.0;
      const double* v = A.f64 + (base - lane_slot) * 9 + lane_slot;
      for (int32_t e = bl; e < len; e += kBL) {
        const int32_t col = next;
        if (e + kBL < len) next = A.col[base + 32 * (int64_t)(e + kBL)];
        double H[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) H[q] = v[(int64_t)e * 288 + 32 * q];
#pragma unroll
        for (int q = 0; q < kR; ++q)
          if (q < nh) {
            const double* xr = p + (r0 + q) * stride + 3 * (int64_t)col;
            const double x0 = xr[0], x1 = xr[1], x2 = xr[2];
#pragma unroll
            for (int j = 0; j < 3; ++j)
              y[3 * q + j] = fma(H[3 * j + 2], x2, fma(H[3 * j + 1], x1, fma(H[3 * j], x0, y[3 * q + j])));
          }
      }
#pragma unroll
      for (int o = kBL / 2; o > 1; o >>= 1)
#pragma unroll
        for (int q = 0; q < kR * 3; ++q) y[q] += __shfl_xor_sync(kFull, y[q], o, kBL);
      if (kHalves)
#pragma unroll
        for (int q = 0; q < kH * 3; ++q) {
          const double hi = q + 3 * kH < 3 * kR ? y[q + 3 * kH] : 0.0;
          const double other = __shfl_xor_sync(kFull, up ? y[q] : hi, 1, kBL);
          y[q] = (up ? hi : y[q]) + other;
        }
    }
    if (in && holds) {
#pragma unroll
      for (int q = 0; q < kH; ++q)
        if (q0 + q < nh) {
          const int64_t o = (r0 + q0 + q) * stride + 3 * (int64_t)row;
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            Ap[o + j] = y[3 * q + j];
            dot[q] = fma(p[o + j], y[3 * q + j], dot[q]);
          }
        }
    }
  }
  let_next_kernel_launch();
  __shared__ double red[kThreads / 32][8];
#pragma unroll
  for (int q = 0; q < kH; ++q) {
#pragma unroll
    for (int o = G; o < 32; o <<= 1) dot[q] += __shfl_xor_sync(kFull, dot[q], o);
    if (lane < G && holds && q0 + q < kR) red[w][r0 + q0 + q] = dot[q];
  }
  __syncthreads();
  if ((int)threadIdx.x < nrhs) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < kThreads / 32; ++i) v += red[i][threadIdx.x];
    pap.sum[threadIdx.x * pap.pitch + blockIdx.x] = v;
  }
}

// Lanes per row by size.  The large-system shapes give each lane two
// right-hand sides and the whole row (64^3, 8 RHS: 0.19 ms; 2 lanes sharing the
// blocks of 8 RHS: 0.23 ms); where the rows do not fill the GPU, 2 or 4 lanes
// share a row's blocks, and more only shorten the sums of a lane to two blocks.
// Whole solves with the lanes of this rule / twice as many / half as many: 45^3,
// 1 RHS (2) 2.87 / - / 3.08 ms; 40^3, 4 RHS (2) 41.8 / - / 42.7; 32^3, 1 RHS,
// five Newton steps (2) 26.5 / 26.7 / -; 20^3, 2 RHS (4) 13.3 / 14.4 / -.
// With five or seven right-hand sides in a lane the blocks are two to an SM and 1 lane
// leaves the last round empty for longer: 50^3, 5 RHS 9.1 ms with 1, 8.0 with 2; 64^3
// 12.6 and 13.6.
// (Loading an entry one ahead of its use: 45^3 2.87 ms as well, 20^3 13.9.)
// A row coupled to very many nodes holds up the whole product, 0.4 to 0.9 us an entry
// and lane, so four lanes share the rows where the longest is beyond kHubRow; below it
// the other rows' sums cost more.  24 iterations at 64^3, 4 RHS, FP64, with one row of
// 327 / 627 / 3,027 blocks, 1 lane and 4: 18.5 / 27.6 / 100 and 14.1 / 16.1 / 32.7 ms
// (15.4 with one lane and a row of 227); 40^3, 1 RHS, 3,027: 2 lanes 31.2, 4 17.5.
// The FP64 product of 3, 5 and 7 right-hand sides in a lane goes out in blocks of 128
// threads, twice as many, where a block has few chunks: the last round is then better
// shared.  FP64 row product, FP32 preconditioner, 256 / 128 threads: 6 RHS (2 x 3) 50^3
// 9.2 / 8.7 ms, 60^3 14.0 / 13.3, 64^3 15.0 / 15.1, 76^3 22.8 / 23.9; 7 RHS, 2 lanes,
// 44^3 7.6 / 7.1, 53^3 12.2 / 11.7, 56^3 12.7 / 12.7, 60^3 14.8 / 15.1; 1 lane 64^3
// 16.1 / 17.9.
constexpr int32_t kHubRow = 192;
template <bool kFF, int kRL, int kR>
static int launch_spmv(gs_ctx ctx, gs_mat m, const float2* xs, const double* p, double* Ap, int nrhs,
                       const PcgScalars* s, Partials& pap) {
  const Sliced A{m->row_order, m->sl_ptr, m->sl_len, m->sl_col, m->sl_ff, m->sl_f64, m->n};
  const int64_t rows = (int64_t)m->n * kRL, sms = std::max(ctx->sm_count, 1);
  const int bl = rows * 4 <= sms * 512 || m->sl_longest > kHubRow ? 4 : (rows * 2 <= sms * (kR > 3 ? 3072 : 2048) ? 2 : 1);
  constexpr int kMin = kR > 3 ? 2 : (kFF && kR < 3 ? 4 : 3);
  auto go = [&](auto kernel, int threads, int per_sm) {
    const int64_t chunks = (rows * bl + threads - 1) / threads;
    pap.n = (int)std::max<int64_t>(1, std::min<int64_t>({chunks, per_sm * sms, (int64_t)kMaxRedBlocks}));
    return launch_chained(ctx, (int64_t)m->n * nrhs, kernel, dim3(pap.n), dim3(threads), 0, A, m->ff_k, xs, p, Ap,
                          3LL * m->n, nrhs, s, pap);
  };
  cudaError_t e = cudaSuccess;
  if constexpr (!kFF && kR >= 3) {
    const bool few = rows * bl <= sms * (kR > 3 ? 2048 : 3072);  // lanes in all
    if (few && bl == 2) {
      GS_CUDA(go(k_pcg_spmv<kFF, 2, kRL, kR, kT / 2, 2 * kMin>, kT / 2, 2 * kMin));
      return GS_OK;
    }
    if constexpr (kR == 3)
      if (few && bl == 1) {
        GS_CUDA(go(k_pcg_spmv<kFF, 1, kRL, kR, kT / 2, 2 * kMin>, kT / 2, 2 * kMin));
        return GS_OK;
      }
  }
  switch (bl) {
    case 1: e = go(k_pcg_spmv<kFF, 1, kRL, kR, kT, kMin>, kT, kMin); break;
    case 2: e = go(k_pcg_spmv<kFF, 2, kRL, kR, kT, kMin>, kT, kMin); break;
    default: e = go(k_pcg_spmv<kFF, 4, kRL, kR, kT, kMin>, kT, kMin); break;
  }
  GS_CUDA(e);
  return GS_OK;
}

template <bool kFF>
static int launch_spmv_rhs(gs_ctx ctx, gs_mat m, const float2* xs, const double* p, double* Ap, int nrhs,
                           const PcgScalars* s, Partials& pap) {
  if (nrhs == 1) return launch_spmv<kFF, 1, 1>(ctx, m, xs, p, Ap, nrhs, s, pap);
  if (nrhs == 2) return launch_spmv<kFF, 2, 1>(ctx, m, xs, p, Ap, nrhs, s, pap);
  // Odd counts and 6 leave places of 2 x 2 or 4 x 2 empty, and an instruction costs the
  // same for a lane without a right-hand side: other shares, but not on systems so
  // small that lanes are what is missing (12^3, 5 RHS: 1.1 ms with 4 lanes of 2, 1.2
  // with 2 of 3), nor where 7 in one lane leave too few (32^3: 3.4 and 3.7 ms; 34^3 4.3
  // and 3.9).  24 iterations at 64^3, FP32 preconditioner, with the shares of 4 and 8 /
  // these / the former product: row 3 RHS 10.7 / 9.8 / 10.5 ms, 5 17.5 / 12.6 / 13.6, 6
  // 17.8 / 15.0 / 15.2, 7 18.2 / 16.0 / 17.0; float-float 3 RHS 7.6 / 7.1 / 9.0, 5 10.9 /
  // 9.3 / 10.5, 6 10.7 / 9.9 / 11.0.  Row product, 53^3: 5 RHS 8.9 (former 9.6), 6 10.6
  // (10.7), 7 11.7 (11.7).
  if (m->n >= 4096) {
    if (kFF) {
      if (nrhs == 3) return launch_spmv<true, 1, 3>(ctx, m, xs, p, Ap, nrhs, s, pap);
      if (nrhs == 5 || nrhs == 6) return launch_spmv<true, 2, 3>(ctx, m, xs, p, Ap, nrhs, s, pap);
    } else {
      if (nrhs == 3) return launch_spmv<false, 1, 3>(ctx, m, xs, p, Ap, nrhs, s, pap);
      if (nrhs == 5) return launch_spmv<false, 1, 5>(ctx, m, xs, p, Ap, nrhs, s, pap);
      if (nrhs == 6) return launch_spmv<false, 2, 3>(ctx, m, xs, p, Ap, nrhs, s, pap);
      if (nrhs == 7 && m->n > 256LL * ctx->sm_count) return launch_spmv<false, 1, 7>(ctx, m, xs, p, Ap, nrhs, s, pap);
    }
  }
  if (nrhs <= 4) return launch_spmv<kFF, 2, 2>(ctx, m, xs, p, Ap, nrhs, s, pap);
  return launch_spmv<kFF, 4, 2>(ctx, m, xs, p, Ap, nrhs, s, pap);
}

// Ap = A p and the partial sums of p . Ap (pap.n is set), at most 8 right-hand
// sides, over the sliced matrix (ensure_sliced); ps: the split operand
// (float-float product) or null (FP64 product).
int pcg_spmv_dot(gs_ctx ctx, gs_mat m, const float2* ps, const double* p, double* Ap, int nrhs, const PcgScalars* s,
                 Partials& pap) {
  GS_PROF(ctx, GS_K_SPMV);
  return ps ? launch_spmv_rhs<true>(ctx, m, ps, p, Ap, nrhs, s, pap)
            : launch_spmv_rhs<false>(ctx, m, nullptr, p, Ap, nrhs, s, pap);
}

// ---------------------------------------------------------------- x, r, ||r||^2, level-1 sums
// A warp takes a level-0 domain and kR right-hand sides: its 3N values of each
// in three passes (lanes along the domain's nodes in slot order, so
// neighbouring lanes read neighbouring entries), r kept in shared memory for
// the sums over the domain's level-1 items.  kR = 2: two right-hand sides'
// loads are in flight together, and more per warp leave too few warps (40^3,
// 4 RHS: 129 us per iteration with four, 122 with two).  What does not come from the kernel just
// before (x, r, p and the domain tables) is loaded before that one has ended.
constexpr int kPitch = 99;  // doubles per right-hand side: 3 N <= 96, spread over the banks

template <int kR>
__global__ void __launch_bounds__(kT, 3) k_pcg_xr(double* __restrict__ x, double* __restrict__ r,
                                                  const double* p, const double* Ap, int64_t stride, int nrhs,
                                                  const int32_t* __restrict__ remap0,
                                                  int32_t n_dom, int N, const int32_t* __restrict__ item1,
                                                  int64_t off1, double* __restrict__ rl, int64_t lstride,
                                                  PcgScalars* s, Partials pap, Partials rrp, int parity) {
  __shared__ double sm_all[kWarps * kR * kPitch];
  __shared__ double s_alpha[kR];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int kb = blockIdx.y * kR;
  double* sm = sm_all + w * (kR * kPitch);
  double rr[kR], rv[kR][3], pv[kR][3], xv[kR][3];
  int64_t o[3];  // this lane's three entries (-1: padding)
  int32_t node = -1, c1 = -1;
  auto load = [&](int32_t d) {
    node = lane < N ? remap0[(int64_t)d * N + lane] : -1;
    c1 = node >= 0 && item1 ? item1[node] : -1;
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int v = t * 32 + lane;
      const int32_t nd = __shfl_sync(kFull, node, v / 3);
      o[t] = v < 3 * N && nd >= 0 ? 3 * (int64_t)nd + v % 3 : -1;
    }
#pragma unroll
    for (int k = 0; k < kR; ++k)
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        const int64_t at = (kb + k) * stride + o[t];
        rv[k][t] = pv[k][t] = xv[k][t] = 0.0;
        if (kb + k < nrhs && o[t] >= 0) rv[k][t] = r[at], pv[k][t] = p[at], xv[k][t] = x[at];
      }
  };
  int32_t d = blockIdx.x * kWarps + w;
  if (s->all_conv) return;  // the product did not write it
  if (d < n_dom) load(d);
  wait_for_previous_kernel();
  if (w < kR && kb + w < nrhs) {
    const int k = kb + w;
    const double sum = warp_sum_partials(pap, k);
    if (lane == 0) {
      s_alpha[w] = take_alpha(s, k, sum, parity, blockIdx.x == 0);
      if (blockIdx.x == 0) s->fp[parity ^ 1][k] = kExpNone;  // k_pcg_p gathers there
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kR; ++k) rr[k] = 0.0;
  while (d < n_dom) {
    double av[kR][3], al[kR];
#pragma unroll
    for (int k = 0; k < kR; ++k) {
      al[k] = kb + k < nrhs ? s_alpha[k] : 0.0;
#pragma unroll
      for (int t = 0; t < 3; ++t) av[k][t] = al[k] != 0.0 && o[t] >= 0 ? Ap[(kb + k) * stride + o[t]] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kR; ++k)
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        if (al[k] != 0.0 && o[t] >= 0) {
          const int64_t at = (kb + k) * stride + o[t];
          x[at] = fma(al[k], pv[k][t], xv[k][t]);
          rv[k][t] = fma(-al[k], av[k][t], rv[k][t]);
          r[at] = rv[k][t];
        }
        rr[k] = fma(rv[k][t], rv[k][t], rr[k]);
        if (item1) sm[k * kPitch + t * 32 + lane] = rv[k][t];
      }
    if (item1) {
      __syncwarp();
      // value c of RHS k summed over each group's slots by kParts lanes, 32 /
      // kParts neighbouring slots each, then the parts (an addition costs the
      // FP64 pipe the same for 3 lanes as for 32)
      constexpr int kV = 3 * kR, kParts = kR == 1 ? 8 : 4, kS = 32 / kParts;
      const int part = lane / kV, kc = lane % kV, k = kc / 3, c = kc % 3;
      const bool act = part < kParts;  // 24 lanes
      const double* mine = sm + (act ? k : 0) * kPitch + c + 3 * kS * (act ? part : 0);
      for (uint32_t left = __ballot_sync(kFull, node >= 0); left;) {
        const int lead = __ffs(left) - 1;
        const int32_t cc = __shfl_sync(kFull, c1, lead);
        const uint32_t g = __ballot_sync(kFull, node >= 0 && c1 == cc);
        double sum = 0.0;
        if (g == 0xffffffffu) {  // the usual domain: full, one item
          double q4[4];
#pragma unroll
          for (int q = 0; q < kS; ++q) q4[q % 4] = q < 4 ? mine[3 * q] : q4[q % 4] + mine[3 * q];
          sum = (q4[0] + q4[1]) + (q4[2] + q4[3]);
        } else {
          const uint32_t gm = (g >> (act ? part * kS : 0)) & ((1u << kS) - 1u);
          for (uint32_t m = act ? gm : 0u; m; m &= m - 1) sum += mine[3 * (__ffs(m) - 1)];
          __syncwarp();
        }
#pragma unroll
        for (int h = kParts / 2; h > 0; h /= 2) sum += __shfl_down_sync(kFull, sum, h * kV);
        if (part == 0 && kb + k < nrhs) rl[(kb + k) * lstride + c + 3 * (off1 + cc)] = sum;
        left &= ~g;
      }
      __syncwarp();
    }
    d += gridDim.x * kWarps;
    if (d < n_dom) load(d);
  }
  let_next_kernel_launch();
  __shared__ double red[kWarps][kR];
  const int ks = sum_index<kR>(lane);
  const double v = warp_sums<kR>(rr, lane);
  if (lane < kR) red[w][ks] = v;
  __syncthreads();
  if ((int)threadIdx.x < kR && kb + (int)threadIdx.x < nrhs) {
    double t = 0.0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) t += red[i][threadIdx.x];
    rrp.sum[(kb + threadIdx.x) * rrp.pitch + blockIdx.x] = t;
  }
}

// x += alpha p, r -= alpha Ap, partial sums of ||r||^2 (rrp.n is set), and rl =
// level-1 sums of r (where the preconditioner has a level 1), at most 8
// right-hand sides.
int pcg_update_xr(gs_ctx ctx, gs_mas mas, double* x, double* r, const double* p, const double* Ap, int nrhs, double* rl,
                  int64_t lstride, PcgScalars* s, const Partials& pap, Partials& rrp, int parity) {
  GS_PROF(ctx, GS_K_PCG_VECTOR);
  const int kr = nrhs == 1 ? 1 : 2;
  // a domain per warp while the partial sums allow it: one wave of longer
  // blocks left a third of the last round empty
  rrp.n = std::max(1, std::min(ceil_div(mas->n_domains[0], kWarps), kMaxRedBlocks));
  const bool coarse = mas->L > 1;
  GS_CUDA(launch_chained(ctx, (int64_t)mas->n * nrhs, kr == 1 ? k_pcg_xr<1> : k_pcg_xr<2>,
                         dim3(rrp.n, ceil_div(nrhs, kr)), dim3(kT), 0, x, r, p, Ap, 3LL * mas->n, nrhs, mas->remap0,
                         mas->n_domains[0], mas->N, coarse ? mas->coarse[1] : nullptr, coarse ? mas->vec_off[1] : 0,
                         rl, lstride, s, pap, rrp, parity));
  return GS_OK;
}

// ---------------------------------------------------------------- p = z + beta p
// Block (g, k): the convergence test of RHS k and its beta from the partial
// sums, then its share of p.  kFF: also the float-float operand of the next
// product, ps = split(p 2^(k_node - K - F)) with 2^F above |p| from the bounds
// |z| < 2^fz, |p_old| < 2^fp, |beta| < 2^eb as max(fz, fp + eb) + 1, node-major
// across right-hand sides; the new p's bound gathers in the other parity's fp.
// A converged RHS keeps p, ps and its bounds.
template <bool kFF>
__global__ void __launch_bounds__(kT) k_pcg_p(double* __restrict__ p, const double* z,
                                              float2* __restrict__ ps, const int32_t* __restrict__ kk, int64_t len,
                                              int nrhs, PcgScalars* s, Partials rrp, Partials rzp, double tol2,
                                              int parity) {
  constexpr int kUnroll = 4;  // strided elements per thread and pass, loaded before they are used
  __shared__ double s_beta;
  __shared__ int s_ex[2], s_stop;
  const int k = blockIdx.y;
  const bool record = blockIdx.x == 0 && threadIdx.x == 0;
  const int64_t o = (int64_t)k * len, step = (int64_t)gridDim.x * kT * kUnroll;
  int64_t i = (int64_t)blockIdx.x * kT * kUnroll + threadIdx.x;
  // p and ||r||^2 do not come from the kernel just before
  double pv[kUnroll];
#pragma unroll
  for (int u = 0; u < kUnroll; ++u) pv[u] = i + u * kT < len ? p[o + i + u * kT] : 0.0;
  double rr = 0.0;
  if (threadIdx.x < 32) rr = warp_sum_partials(rrp, k);
  wait_for_previous_kernel();
  // all_conv is read once for the block: this grid's recording blocks may set it
  double rz = 0.0;
  bool over = false;
  if (threadIdx.x < 32) {
    over = __shfl_sync(kFull, threadIdx.x == 0 ? s->all_conv : 0, 0) != 0;
    if (!over) rz = warp_sum_partials(rzp, k);
  }
  if (threadIdx.x == 0) {
    s_ex[0] = s_ex[1] = kExpNone;
    s_stop = over || test_convergence(s, k, rr, tol2, record);
    s_beta = rz / s->rz[parity][k];
  }
  int ex = kExpNone;
  if (kFF)
    for (int g = threadIdx.x; g < rzp.n; g += kT) ex = max(ex, __ldcg(rzp.ex + (size_t)k * rzp.pitch + g));
  __syncthreads();
  if (s_stop) {
    if (kFF && record) atomicMax(&s->fp[parity ^ 1][k], s->fp[parity][k]);
    return;
  }
  const double be = s_beta;
  if (record) {
    s->rz[parity ^ 1][k] = rz;
    if (!isfinite(rz)) {
      atomicOr(&s->flags, kErrNonFinite);
      s->bad[k] = 1;
    }
  }
  int F = 0;
  if (kFF) {
    ex = __reduce_max_sync(kFull, ex);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_ex[0], ex);
    __syncthreads();
    const int eb = ex_bound(be), fp = s->fp[parity][k];
    const int fb = (fp == kExpNone || eb == kExpNone) ? kExpNone : fp + eb;
    const int fmax = max(s_ex[0], fb);
    F = fmax == kExpNone ? 0 : fmax + 1;
    if (record) s->fsplit[k] = F;
    ex = kExpNone;
  }
  while (i < len) {
    double zv[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) zv[u] = i + u * kT < len ? z[o + i + u * kT] : 0.0;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int64_t j = i + u * kT;
      if (j < len) {
        const double v = fma(be, pv[u], zv[u]);
        p[o + j] = v;
        if (kFF) {
          ex = max(ex, ex_bound(v));
          const uint32_t node = (uint32_t)j / 3u;
          ps[((int64_t)node * nrhs + k) * 3 + ((uint32_t)j - 3u * node)] = ff_split_bits(v, kk[node] - F);
        }
      }
    }
    i += step;
    if (i >= len) break;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) pv[u] = i + u * kT < len ? p[o + i + u * kT] : 0.0;
  }
  let_next_kernel_launch();
  if (kFF) {
    ex = __reduce_max_sync(kFull, ex);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_ex[1], ex);
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(&s->fp[parity ^ 1][k], s_ex[1]);
  }
}

// Folds the partial sums of a reduction over very many domains to 64 per RHS.
constexpr int kFold = 64;
__global__ void __launch_bounds__(kT) k_fold(Partials a, Partials out, const int* skip) {
  wait_for_previous_kernel();
  if (*skip) return;
  const int k = blockIdx.y, per = (a.n + kFold - 1) / kFold, g0 = blockIdx.x * per;
  Partials mine = a;
  mine.sum += g0;
  mine.n = max(0, min(per, a.n - g0));
  const double v = threadIdx.x < 32 ? warp_sum_partials(mine, k) : 0.0;
  __shared__ int s_ex;
  if (threadIdx.x == 0) s_ex = kExpNone;
  __syncthreads();
  int e = kExpNone;
  for (int g = threadIdx.x; g < mine.n; g += kT) e = max(e, a.ex[(size_t)k * a.pitch + g0 + g]);
  e = __reduce_max_sync(kFull, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_ex, e);
  __syncthreads();
  if (threadIdx.x == 0) {
    out.sum[k * out.pitch + blockIdx.x] = v;
    out.ex[k * out.pitch + blockIdx.x] = s_ex;
  }
}

// The convergence test, beta and p = z + beta p from the partial sums of
// ||r||^2 and r . z; fold: room for kFold partials per right-hand side.
int pcg_update_p(gs_ctx ctx, gs_mat m, double* p, const double* z, float2* ps, int nrhs, PcgScalars* s,
                 const Partials& rrp, const Partials& rzp, Partials fold, double tol2, int parity) {
  GS_PROF(ctx, GS_K_PCG_VECTOR);
  const int64_t len = 3LL * m->n, work = (int64_t)m->n * nrhs;
  Partials rz = rzp;
  if (rzp.n > kMaxRedBlocks) {  // every block below would read them all
    GS_CUDA(launch_chained(ctx, work, k_fold, dim3(kFold, nrhs), dim3(kT), 0, rzp, fold, &s->all_conv));
    rz = fold;
    rz.n = kFold;
  }
  // blocks per SM over all right-hand sides: each first adds the partial sums,
  // so few and long ones where there is much to do (64^3, 8 RHS, 24 iterations:
  // 2 per SM 13.5 ms, 4 13.1, 6 and 8 13.4, 24 13.8), and eight where the chain of
  // loads of a block is all there is (40^3, 4 RHS: 8 40.8 ms, 4 41.3)
  const int gx = (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(len, kT * 4),
                                                             ((work > kSmallWork ? 4LL : 8LL) * std::max(ctx->sm_count, 1) + nrhs - 1) / nrhs));
  GS_CUDA(launch_chained(ctx, work, ps ? k_pcg_p<true> : k_pcg_p<false>, dim3(gx, nrhs), dim3(kT), 0, p, z, ps,
                         ps ? m->ff_k : nullptr, len, nrhs, s, rrp, rz, tol2, parity));
  return GS_OK;
}

}  // namespace gs
