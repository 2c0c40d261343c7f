// Level-0 MAS product in FP64 accuracy on the F16 tensor cores (Eq. 6 at
// level 0), by exact integer splitting of both operands (the Ozaki scheme).
//
// FP64 FMA runs at 2 per clock per SM on this part, so the FP64 dense
// product z_d = M_d^{-1} r_d is bound by the FP64 pipe.  Here both operands
// become sums of small integers times powers of two, every partial product
// is exact in the tensor core's FP32 accumulator, and only a short integer
// combination remains per output:
//   * build time: row i of M_d^{-1} gets an exponent a_i with |M_ik| < 2^(a_i-1);
//     X_ik = rint(M_ik 2^(56-a_i)) (|X| < 2^55) is cut into 7 balanced base-256
//     digits m^(1..7) in [-128, 127] (X = sum_p m^(p) 256^(7-p)), stored as the
//     bytes m + 128 (a row whose leading digit would be 128 takes a_i + 1);
//   * apply: column k of r_d gets b_k with |r_jk| < 2^(b_k-1), likewise
//     Y_jk = rint(r_jk 2^(56-b_k)) -> digits n^(1..7) in [-128, 128];
//   * G_s = sum_{p+q=s} m^(p) n^(q) for s = 2..9 (products of digits <= 2^14,
//     96 terms, <= 7 pairs: |G_s| < 2^24, exact in FP32): the B operand holds
//     all 7 digit columns of r (plus a zero one), so one MMA per digit matrix
//     and K step writes the groups p+2 .. 9 into TMEM columns 8p .. 63 (one more
//     group, not read, where N is rounded up to a multiple of 16); each G_s
//     collects in its own 8 columns;
//   * z_ik = 2^(a_i + b_k - 72) sum_{s=2..9} G_s 256^(9-s), combined in
//     64-bit integers (two halves) and rounded once to a double in integer
//     arithmetic, so the epilogue spends one FP64 add (the coarse levels).
// The roundings of X and Y move z_ik by at most 2^(a_i - 57) sum_j |r_jk| + 2^(b_k - 57)
// sum_j |M_ij|, half a unit of each operand against the other, and the dropped terms
// (p + q > 9) by 2^(a_i + b_k - 57): within the bound of the sum in FP64, 96 2^-53 of
// the row's and column's largest, and 96 2^-57 of 2^(a_i + b_k) altogether.
//
// One CTA of 256 threads per domain.  The digit bytes come into a shared-memory
// ring by bulk asynchronous copies; two threads per row read them, expand them
// to F16 (a byte permute and a subtraction for two entries) and store them to
// TMEM as the MMA's A operand.  What bounds it: no longer the bytes (7 per entry;
// BF16 digits, copied to shared memory as they lay, were 14, and 81 % of the
// DRAM rate) but the chain of steps within a domain, about 16000 clocks with
// four domains to an SM, half of it the seven digits.  With r . z, 45^3, 1 RHS:
// 74 -> 51 us; 24 bodies, 1 RHS: 140 -> 99; 64^3, 8 RHS: 214 -> 172 without it.
// Tried: digits prefetched into registers (57 us at 45^3, against 48 of the same
// without r . z), three A operands and two CTAs per SM (70).  All waits are
// bounded (kErrTimeout); TMEM is always freed.
#include <algorithm>

#include "common.cuh"
#include "fp64split.cuh"
#include "pcg_state.cuh"
#include "umma.cuh"

namespace gs {
namespace f64tc {

constexpr int kDigits = 7;
constexpr int kThreads = 256;
constexpr int kM = 128;

// TMEM: groups s = 2..10, 8 columns each, then kBufs A operands of LD / 2 columns.
constexpr int kACol = 80;
__host__ __device__ constexpr int tmem_cols(int bufs, int ld) {
  const int need = kACol + bufs * (ld / 2);
  return need <= 128 ? 128 : (need <= 256 ? 256 : 512);
}
__host__ __device__ constexpr size_t ring_bytes(int slots, int ld) { return 128 + (size_t)slots * ld * ld; }

struct Levels {
  const int32_t* coarse[8];
  const int2* kids[8];  // level l's items as sums of level l - 1's (gs_mas_s::kids), or null
  int64_t vec_off[8];
  int L;
};

// T 2^e as the nearest double (ties to even), T = hi 2^32 + lo with
// |hi|, |lo| < 2^49.
__device__ __forceinline__ double scaled_to_double(long long hi, long long lo, int e) {
  return combine_to_double(hi, lo, 32, e);
}

// kCoarse = false: level-0 domains, r gathered through remap0, z = level-0
//   product + prolongated coarse results, written per node; kDot: also the
//   domain's part of r . z per right-hand side and the exponent bound of its z;
// kCoarse = true: coarse-level domains (job tables), r and z are the level's
//   contiguous multilevel vectors rl, zl; a level with al.kids gathers its r
//   as the sums of its items' children of the level below.
// kSlots: digits in the ring; kBufs: A operands in TMEM (a digit is stored while
// the MMAs of the kBufs - 1 before it run); kCtas of them per SM.
// Roles after the operand B is written: the warps that own rows of TMEM lanes
// 0 .. LD - 1 expand and store the digits and later take the results, warp 3
// issues the MMAs and the copies, warp 7 sums the prolongated coarse results.  r . z costs a
// CTA ten FP64 instructions per warp (warp_sums), the separate pass it replaces
// 9 us at 45^3.
template <bool kCoarse, bool kDot, int kSlots, int kBufs, int kCtas, int LD>
__global__ void __launch_bounds__(kThreads, kCtas) k_level0_f64tc(
    const uint8_t* const* __restrict__ dig_tab, const int32_t* const* __restrict__ exp_tab,
    const int32_t* __restrict__ job_level, const int32_t* __restrict__ job_dom, const int32_t* __restrict__ remap0,
    int N, int nrhs, Levels al, const double* r, int64_t stride, const double* zl, int64_t lstride,
    double* __restrict__ z, int* __restrict__ flags, const int* skip, Partials dot) {
  using namespace umma;
  // The digits may be copied before the kernel ahead has ended where that is the
  // restriction or the coarse product: it wrote neither them nor *skip.
  constexpr bool kEarly = kCoarse || kDot;
  if (!kEarly) wait_for_previous_kernel();
  constexpr int ld = LD;  // 3 N
  constexpr int kPer = (8 * LD + kThreads - 1) / kThreads;  // entries of r per thread: e = tid + m kThreads = k ld + j
  constexpr int kChunks = LD / 16, kHalf = (kChunks + 1) / 2, kRowWarps = (LD + 31) / 32;
  __shared__ __align__(128) unsigned char sB[LD / 8 * 1024];  // 4 pair operands [n^(2j+1) | n^(2j+2)]
  __shared__ double sr[kDot ? 8 * LD : 1];                     // r, for r . z
  __shared__ double scoarse[kCoarse ? 1 : 8 * LD];
  __shared__ int32_t snode[32];  // node of every slot of the domain (-1: padding)
  __shared__ int sexp[8];        // biased exponent maxima of the RHS columns
  __shared__ uint64_t full[kSlots], ready[kBufs], freed[kBufs], drained, summed;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  constexpr uint32_t dig_bytes = LD * LD, kCols = tmem_cols(kBufs, LD);
  __shared__ uint32_t tslot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // loads that depend on nothing leave together
  const int lvl = kCoarse ? job_level[blockIdx.x] : 0;
  const int32_t d = kCoarse ? job_dom[blockIdx.x] : (int32_t)blockIdx.x;
  const uint8_t* dd = dig_tab[lvl] + (int64_t)d * kDigits * LD * LD;
  int32_t node_of[kPer];  // nodes of this thread's entries of r; coarse: their children's lane masks
  int32_t first_of[kPer];
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int e = tid + m * kThreads;
    const bool in = e / ld < nrhs && e < 8 * ld;
    node_of[m] = kCoarse ? 0 : (in ? remap0[(int64_t)d * N + e % ld / 3] : -1);
    first_of[m] = 0;
    if (kCoarse && in && al.kids[lvl]) {
      const int2 kid = al.kids[lvl][(int64_t)d * N + e % ld / 3];
      first_of[m] = kid.x, node_of[m] = kid.y;
    }
  }
  const int32_t my_node = kCoarse ? 0 : remap0[(int64_t)d * N + min(lane, N - 1)];
  if (skip && *skip) return;  // whole CTA, before any barrier or TMEM use
  const int64_t cbase = kCoarse ? 3 * (al.vec_off[lvl] + (int64_t)d * N) : 0;  // coarse: first entry of the domain
  // Warps w and w + 4 share TMEM lane quarter w % 4: they expand half a row
  // each and take the right-hand sides 0..3 and 4..7 of its results.
  constexpr int kRpt = 4;  // right-hand sides per epilogue thread
  const int q4 = warp & 3, half = warp >> 2, k0 = half * kRpt;
  const int i_row = q4 * 32 + lane;
  const bool rows = q4 < kRowWarps;  // whole warp

  if (tid == 0) {
    for (int q = 0; q < kSlots; ++q) mbar_init(&full[q], 1);
    for (int q = 0; q < kBufs; ++q) mbar_init(&freed[q], 1), mbar_init(&ready[q], 2 * kRowWarps);
    mbar_init(&drained, 1);
    mbar_init(&summed, 1);
    fence_mbar_init();
    for (int q = 0; q < kSlots; ++q) {
      mbar_arrive_expect_tx(&full[q], dig_bytes);
      bulk_g2s(ring + q * dig_bytes, dd + q * dig_bytes, dig_bytes, &full[q]);
    }
  }
  if (tid < 8) sexp[tid] = 0;
  if (tid < 32) snode[tid] = tid < N ? my_node : -1;
  if (warp == 0) {
    tmem_alloc(&tslot, kCols);
    tmem_relinquish();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = tslot;
  if (kEarly) wait_for_previous_kernel();
  // Digit p of this thread's half row, chunk c (16 entries) at [c][row] of its
  // slot, to the A operand: false where a wait gave up.
  bool ok = true;
  auto store_digit = [&](int p) {
    const unsigned char* mine = ring + (p % kSlots) * dig_bytes + (half * kHalf * ld + min(i_row, ld - 1)) * 16;
    const uint32_t ta = tmem + ((uint32_t)(q4 * 32) << 16) + kACol + half * kHalf * 8 + (p % kBufs) * (ld / 2);
    ok = ok && mbar_wait(&full[p % kSlots], (uint32_t)(p / kSlots) & 1u);
    uint32_t v[kHalf][8];  // expanded while the MMAs of the digit before still read the operand
#pragma unroll
    for (int j = 0; j < kHalf; ++j)
      if (half * kHalf + j < kChunks) {  // whole warp
        const uint4 b = *reinterpret_cast<const uint4*>(mine + j * ld * 16);
        expand_digit_bytes(b.x, v[j][0], v[j][1]);
        expand_digit_bytes(b.y, v[j][2], v[j][3]);
        expand_digit_bytes(b.z, v[j][4], v[j][5]);
        expand_digit_bytes(b.w, v[j][6], v[j][7]);
      }
    if (p >= kBufs) ok = ok && mbar_wait(&freed[p % kBufs], (uint32_t)(p / kBufs - 1) & 1u);
    ok = __all_sync(kFull, ok);
    if (!ok) return false;
    fence_after_sync();
#pragma unroll
    for (int j = 0; j < kHalf; ++j)
      if (half * kHalf + j < kChunks) tmem_st_32x32b_x8(ta + 8 * j, v[j]);
    tmem_wait_st();
    fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive(&ready[p % kBufs]);
    return true;
  };
  // r_d once into registers (entry e = k * ld + j), column exponents by
  // shared-memory atomics, then the digits into the four pair operands
  double rv[kPer];
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int e = tid + m * kThreads;
    const int k = e / ld, j = e - k * ld;
    rv[m] = 0.0;
    if (k < nrhs && k < 8) {
      if (kCoarse) {
        if (al.kids[lvl]) {
          const double* rk = r + k * lstride + 3 * (al.vec_off[lvl - 1] + first_of[m]) + j % 3;
          rv[m] = sum_children(rk, (uint32_t)node_of[m]);
        } else {
          rv[m] = r[k * lstride + cbase + j];
        }
      } else if (node_of[m] >= 0) {
        rv[m] = r[k * stride + 3 * (int64_t)node_of[m] + j % 3];
      }
    }
  }
  if (rows) store_digit(0);  // while r is on its way
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int e = tid + m * kThreads;
    const int k = e / ld;
    if (k >= nrhs || k >= 8) continue;
    if (kDot) sr[e] = rv[m];
    int eb = biased_exp(rv[m]);  // integer test: no FP64 compare
    if (LD % 32 == 0) {          // one right-hand side per warp
      eb = __reduce_max_sync(kFull, eb);
      if (lane == 0) atomicMax(&sexp[k], eb);
    } else if (eb) {
      atomicMax(&sexp[k], eb);
    }
  }
  __syncthreads();
  // element (n, kk) of a pair operand at (kk/8)*256 + (n/8)*128 + (n%8)*16 + (kk%8)*2
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int e = tid + m * kThreads;
    if (e >= nrhs * ld) break;  // columns of absent right-hand sides stay unset: their results are not read
    const int k = e / ld, j = e - k * ld;
    const long long y = scaled_rint(rv[m], sexp[k] - 1021);  // 0 for zero entries
    // column n = 8 q + k; q = 7: the missing 8th digit, zero
    write_digits256_f16(y, sB + (j >> 3) * 1024 + (j & 7) * 2 + k * 16);
  }
  fence_proxy_async();
  __syncthreads();

  const int32_t node_row = rows && i_row < ld ? snode[i_row / 3] : -1;
  const int c_row = i_row % 3;
  int a_row = -100000;
  if (node_row >= 0) a_row = exp_tab[lvl][(int64_t)d * ld + i_row];
  // one copy of the loops' code where each step waits for the one before anyway:
  // a CTA runs them once, from a cold instruction cache
  constexpr int kUnroll = kBufs == 1 ? 1 : kDigits;
  if (rows) {
#pragma unroll kUnroll
    for (int p = 1; p < kDigits; ++p)
      if (!store_digit(p)) break;
    let_next_kernel_launch();
    constexpr int kLast = kDigits - 1;  // the MMAs end in order
    ok = ok && __all_sync(kFull, mbar_wait(&freed[kLast % kBufs], (uint32_t)(kLast / kBufs) & 1u));
    if (!kCoarse) ok = ok && __all_sync(kFull, mbar_wait(&summed, 0));
    if (!ok && lane == 0) atomicOr(flags, kErrTimeout);
    fence_after_sync();
  } else if (warp == 3) {
    let_next_kernel_launch();
    if (lane == 0) {
      // descriptors are built once; their 14-bit address fields are advanced
      // by adding byte offsets / 16
      const uint64_t db0 = smem_desc(smem_u32(sB), 1024, 128);
      int copied = kSlots;
      bool good = true;
#pragma unroll kUnroll
      for (int p = 0; p < kDigits; ++p) {
        good = good && mbar_wait(&ready[p % kBufs], (uint32_t)(p / kBufs) & 1u);
        if (!good) break;
        fence_after_sync();
        const uint32_t idesc = idesc_f16_f32(kM, (64 - 8 * p + 15) / 16 * 16);
        const uint32_t ta = tmem + kACol + (p % kBufs) * (ld / 2);
#pragma unroll
        for (int ks = 0; ks < kChunks; ++ks)
          mma_f16_ts(tmem + 8u * p, ta + 8u * ks, db0 + ks * (2048u >> 4), idesc, (p > 0 || ks > 0) ? 1u : 0u);
        mma_commit(&freed[p % kBufs]);
        if (p + kSlots < kDigits) {  // every row warp has read this slot
          mbar_arrive_expect_tx(&full[p % kSlots], dig_bytes);
          bulk_g2s(ring + (p % kSlots) * dig_bytes, dd + (p + kSlots) * dig_bytes, dig_bytes, &full[p % kSlots]);
          ++copied;
        }
      }
      if (!good) {  // whatever was issued ends before the CTA leaves
        atomicOr(flags, kErrTimeout);
        mma_commit(&drained);
        mbar_wait(&drained, 0);
        for (int q = 0; q < kSlots; ++q) mbar_wait(&full[q], (uint32_t)((copied - 1 - q) / kSlots) & 1u);
      }
    }
  } else {
    let_next_kernel_launch();
    if (!kCoarse && warp == 7) {
      // the prolongated coarse results, lane s holding slot s's items; the first
      // coarse level assigns: one FP64 add fewer per output
      const int32_t node = lane < N ? snode[lane] : -1;
      int32_t item[8];
#pragma unroll
      for (int l = 1; l < 8; ++l) item[l] = l < al.L && node >= 0 ? al.coarse[l][node] : 0;
      constexpr int kU = 6;
      for (int e0 = 0; e0 < nrhs * ld; e0 += 32 * kU) {
        double v[kU];
        int64_t at[kU];
        int slot[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const int e = min(e0 + 32 * u + lane, nrhs * ld - 1);
          const int k = e / ld, j = e - k * ld;
          slot[u] = j / 3;
          at[u] = k * lstride + j % 3;
          v[u] = 0.0;
        }
#pragma unroll
        for (int l = 1; l < 8; ++l) {
          if (l >= al.L) break;
          double t[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u)
            t[u] = zl[at[u] + 3 * (al.vec_off[l] + __shfl_sync(kFull, item[l], slot[u]))];
#pragma unroll
          for (int u = 0; u < kU; ++u) v[u] = l == 1 ? t[u] : v[u] + t[u];
        }
#pragma unroll
        for (int u = 0; u < kU; ++u)
          if (e0 + 32 * u + lane < nrhs * ld) scoarse[e0 + 32 * u + lane] = v[u];
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&summed);
    }
  }
  double dacc[kRpt];
  int dex[kRpt];
#pragma unroll
  for (int k = 0; k < kRpt; ++k) dacc[k] = 0.0, dex[k] = kExpNone;
  if (rows && ok && k0 < nrhs) {  // whole warp
    const uint32_t ta = tmem + ((uint32_t)(q4 * 32) << 16);
    float g[8 * kRpt];  // groups s = 2..9 of this thread's RHS: g[kRpt (s - 2) + k]
    tmem_ld_32x32b_8x4(ta + k0, 8, g);
    if (node_row >= 0) {
#pragma unroll
      for (int k = 0; k < kRpt; ++k) {
        const int kk = k0 + k;
        if (kk >= nrhs) break;
        double v = 0.0;
        if (sexp[kk] && a_row > -100000) {
          // T = hi 2^32 + lo, hi = sum_{s=2..5} G_s 256^(5-s), lo = sum_{s=6..9} G_s 256^(9-s)
          long long hi = __float2int_rn(g[3 * kRpt + k]), lo = __float2int_rn(g[7 * kRpt + k]);
#pragma unroll
          for (int s = 0; s < 3; ++s) {
            hi += (long long)__float2int_rn(g[kRpt * s + k]) * (1 << (24 - 8 * s));
            lo += (long long)__float2int_rn(g[kRpt * (s + 4) + k]) * (1 << (24 - 8 * s));
          }
          const int e = a_row + (sexp[kk] - 1021) - 72;  // z = T 2^e, T = hi 2^32 + lo
          if (e < 900) v = scaled_to_double(hi, lo, e);
        }
        if (kCoarse) {
          z[kk * lstride + cbase + i_row] = v;
        } else {
          v += scoarse[kk * ld + i_row];
          z[kk * stride + 3 * (int64_t)node_row + c_row] = v;
          if (kDot) {
            dacc[k] = sr[kk * ld + i_row] * v;
            dex[k] = ex_bound(v);
          }
        }
      }
    }
  }
  __shared__ double red[kThreads / 32][kRpt];
  __shared__ int redx[kThreads / 32][kRpt];
  if (kDot) {
    const bool some = rows && k0 < nrhs;  // whole warp: the others add zeros at the FP64 pipe's full price
    const int k = sum_index<kRpt>(lane);
    const double v = some ? warp_sums<kRpt>(dacc, lane) : 0.0;
#pragma unroll
    for (int q = 0; q < kRpt; ++q) {
      const int e = some ? __reduce_max_sync(kFull, dex[q]) : kExpNone;
      if (lane == 0) redx[warp][q] = e;
    }
    if (lane < kRpt) red[warp][k] = v;
  }
  fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    fence_after_sync();
    tmem_dealloc(tmem, kCols);
  }
  if (kDot && tid < nrhs) {
    double v = 0.0;
    int e = kExpNone;
#pragma unroll
    for (int q = 0; q < kRowWarps; ++q) {
      v += red[tid / kRpt * 4 + q][tid % kRpt];
      e = max(e, redx[tid / kRpt * 4 + q][tid % kRpt]);
    }
    dot.sum[(size_t)tid * dot.pitch + d] = v;
    dot.ex[(size_t)tid * dot.pitch + d] = e;
  }
}

}  // namespace f64tc

// GS_TUNE_F64_TC: 1 / 2 / 4 stream the digit bytes of this file, 3 the
// symmetric digit bytes of mas_apply_f64sym.cu; the storage is made when the
// preconditioner is built for the value set then.
bool level0_f64tc_usable(gs_ctx ctx, gs_mas mas, int nrhs) {
  if (mas->precision != GS_PREC_FP64 || nrhs < 1 || nrhs > 8) return false;
  const int t = ctx->tune[GS_TUNE_F64_TC];
  if (t == 3) return !mas->dig8.empty();
  return (t == 1 || t == 2 || t == 4) && !mas->dig64.empty();
}

int level0_f64tc_alloc(gs_ctx ctx, gs_mas mas) {
  const int ld = 3 * mas->N;
  const int t = ctx->tune[GS_TUNE_F64_TC];
  if (t == 0 || t == 3 || ld % 16 != 0 || ld > f64tc::kM || !mas->dig64.empty()) return GS_OK;
  for (int l = 0; l < mas->L; ++l) {  // every level: level 0 and the coarse levels
    const size_t n_dom = (size_t)std::max(mas->n_domains[l], 1);
    void* dg = nullptr;
    int32_t* ex = nullptr;
    GS_TRY(ctx->alloc(&dg, n_dom * f64tc::kDigits * ld * ld));
    mas->dig64.push_back(dg);
    GS_TRY(ctx->alloc((void**)&ex, n_dom * ld * 4));
    mas->dig64_exp.push_back(ex);
  }
  GS_TRY(ctx->alloc((void**)&mas->d_dig_tab, 16 * sizeof(void*)));
  std::vector<void*> hp(16, nullptr);
  for (int l = 0; l < mas->L; ++l) hp[l] = mas->dig64[l], hp[8 + l] = mas->dig64_exp[l];
  GS_CUDA(cudaMemcpyAsync(mas->d_dig_tab, hp.data(), 16 * sizeof(void*), cudaMemcpyHostToDevice, ctx->stream));
  return GS_OK;
}

int level0_f64tc_prepare(gs_ctx ctx, gs_mas mas) {  // 3: symmetric digit bytes; 1, 2, 4 were cut with the inverses
  if (mas->precision != GS_PREC_FP64 || ctx->tune[GS_TUNE_F64_TC] != 3) return GS_OK;
  return f64sym_shape_ok(mas->N) ? f64sym_prepare(ctx, mas) : GS_OK;
}

static f64tc::Levels f64tc_levels(gs_mas mas) {
  f64tc::Levels al{};
  al.L = mas->L;
  for (int l = 0; l < mas->L; ++l) al.coarse[l] = mas->coarse[l], al.vec_off[l] = mas->vec_off[l];
  return al;
}

template <bool kCoarse, bool kDot, int kSlots, int kBufs, int kCtas, int LD>
static int launch_digits(gs_ctx ctx, gs_mas mas, int nrhs, const f64tc::Levels& al, const double* r, int64_t stride,
                         const double* zl, int64_t lstride, double* z, const int* skip, const Partials& dot) {
  const auto kernel = f64tc::k_level0_f64tc<kCoarse, kDot, kSlots, kBufs, kCtas, LD>;
  const size_t smem = f64tc::ring_bytes(kSlots, LD);
  GS_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int jobs = kCoarse ? mas->n_coarse_jobs : mas->n_domains[0];
  const int32_t* jt = kCoarse ? mas->d_coarse_jobs : nullptr;
  GS_CUDA(launch_chained(ctx, (int64_t)mas->n * nrhs, kernel, dim3(jobs), dim3(f64tc::kThreads), smem,
                         (const uint8_t* const*)mas->d_dig_tab, (const int32_t* const*)(mas->d_dig_tab + 8), jt,
                         jt ? jt + jobs : nullptr, mas->remap0, mas->N, nrhs, al, r, stride, zl, lstride, z,
                         ctx->d_flags, skip, dot));
  return GS_OK;
}

// By the number of domains: where every SM holds one at most, all 7 digits are
// copied at once and each has its own A operand in TMEM, so that no step waits
// for an MMA; where it holds two, 3 operands; else one, and a ring of 3 digits,
// so that four CTAs share an SM.  One operand for the 128 domains of a 16^3 body
// as well: 6.2 against 5.5 ms for its solve.
template <bool kCoarse, bool kDot>
static int launch_digits_shape(gs_ctx ctx, gs_mas mas, int nrhs, const f64tc::Levels& al, const double* r,
                               int64_t stride, const double* zl, int64_t lstride, double* z, const int* skip,
                               const Partials& dot) {
  const int jobs = kCoarse ? mas->n_coarse_jobs : mas->n_domains[0], sms = std::max(ctx->sm_count, 1);
#define GS_DIGITS(S, B, C, LD) \
  launch_digits<kCoarse, kDot, S, B, C, LD>(ctx, mas, nrhs, al, r, stride, zl, lstride, z, skip, dot)
  if (mas->N == 32) {  // 3 N = 96 or 48 (the digit storage is made only for N = 32 and 16)
    if (jobs <= sms) return GS_DIGITS(f64tc::kDigits, f64tc::kDigits, 1, 96);
    if (jobs <= 2 * sms) return GS_DIGITS(f64tc::kDigits, 3, 2, 96);
    return GS_DIGITS(3, 1, 4, 96);
  }
  return jobs <= 2 * sms ? GS_DIGITS(f64tc::kDigits, f64tc::kDigits, 2, 48) : GS_DIGITS(3, 2, 4, 48);
#undef GS_DIGITS
}

int level0_f64tc_launch(gs_ctx ctx, gs_mas mas, int nrhs, const double* r, int64_t stride, const double* zl,
                        int64_t lstride, double* z, const int* skip, const Partials* dot) {
  GS_CHECK(level0_f64tc_usable(ctx, mas, nrhs), GS_ERR_UNSUPPORTED, "FP64 tensor-core apply: not available");
  if (ctx->tune[GS_TUNE_F64_TC] == 3) return f64sym_level0_launch(ctx, mas, nrhs, r, stride, zl, lstride, z, skip);
  if (mas->n_domains[0] == 0) return GS_OK;
  return dot ? launch_digits_shape<false, true>(ctx, mas, nrhs, f64tc_levels(mas), r, stride, zl, lstride, z, skip, *dot)
             : launch_digits_shape<false, false>(ctx, mas, nrhs, f64tc_levels(mas), r, stride, zl, lstride, z, skip,
                                                 Partials{});
}

int coarse_f64tc_launch(gs_ctx ctx, gs_mas mas, int nrhs, const double* rl, double* zl, int64_t lstride,
                        const int* skip, bool from_kids) {
  GS_CHECK(level0_f64tc_usable(ctx, mas, nrhs), GS_ERR_UNSUPPORTED, "FP64 tensor-core apply: not available");
  if (ctx->tune[GS_TUNE_F64_TC] == 3) return f64sym_coarse_launch(ctx, mas, nrhs, rl, zl, lstride, skip);
  if (mas->n_coarse_jobs == 0) return GS_OK;
  f64tc::Levels al = f64tc_levels(mas);
  if (from_kids)
    for (int l = 2; l < mas->L; ++l) al.kids[l] = mas->kids[l];
  return launch_digits_shape<true, false>(ctx, mas, nrhs, al, rl, 0, nullptr, lstride, zl, skip, Partials{});
}

}  // namespace gs
