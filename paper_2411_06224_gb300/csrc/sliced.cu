// Sliced copy of an assembled matrix for PCG's own product (pcg_fused.cu):
// the full symmetric matrix, 32 rows of the row order (longest first within
// windows, spmv.cu) to a slice, entry e of the 32 rows side by side.
//
// The stored form keeps the upper triangle once and reaches the lower one by
// reference, so a warp of a row product reads as many scattered 72-byte blocks
// as it holds rows; its L1 traffic bounded the float-float product (73 % of the
// L1 throughput at 48^3, 8 RHS).  Here the same warp reads 32 (or 8) rows'
// values side by side and knows their addresses before the columns arrive, for
// twice the matrix bytes from DRAM, which that kernel has to spare.  The rows
// are nearly equally long within a slice, so little is padding (never read).
// Values come in the order of the row product: the row's stored blocks, then
// the transposed ones, so the sums keep their order.
#include <algorithm>

#include "common.cuh"
#include "ff.cuh"
#include "primitives.cuh"
#include "sort_scan.cuh"

namespace gs {

int ensure_row_order(gs_ctx ctx, gs_mat m);

// Length of every row of the order, the longest of each slice (a warp per
// slice; one slice more, of length 0, ends the scan) and of all (*longest: 0).
__global__ void k_slice_len(const int32_t* __restrict__ row_order, const int32_t* __restrict__ row_ptr,
                            const int32_t* __restrict__ lo_ptr, int32_t n, int32_t n_slices,
                            int32_t* __restrict__ len, int32_t* __restrict__ most, int32_t* __restrict__ longest) {
  const int32_t t = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x), s = t >> 5;
  if (s > n_slices) return;  // whole warp
  int32_t l = 0;
  if (t < n) {
    const int32_t r = row_order[t];
    l = row_ptr[r + 1] - row_ptr[r] + lo_ptr[r + 1] - lo_ptr[r];
    len[t] = l;
  }
  const int32_t m = __reduce_max_sync(kFull, l);
  if ((t & 31) == 0) {
    most[s] = m;
    if (m > *(volatile int32_t*)longest) atomicMax(longest, m);
  }
}

// Column of every entry, and its stored block (complemented: transposed).  A
// warp per slice.
__global__ void k_slice_entries(const int32_t* __restrict__ row_order, const int32_t* __restrict__ row_ptr,
                                const int32_t* __restrict__ cid, const int32_t* __restrict__ lo_ptr,
                                const int32_t* __restrict__ lo_idx, const int32_t* __restrict__ lo_col, int32_t n,
                                const int32_t* __restrict__ ptr, int32_t* __restrict__ col, int32_t* __restrict__ blk) {
  const int32_t t = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
  if (t >= n) return;
  const int32_t r = row_order[t], u0 = row_ptr[r], nu = row_ptr[r + 1] - u0, l0 = lo_ptr[r], nl = lo_ptr[r + 1] - l0;
  int64_t o = (int64_t)ptr[t >> 5] * 32 + (t & 31);
  for (int32_t e = 0; e < nu; ++e, o += 32) col[o] = cid[u0 + e], blk[o] = u0 + e;
  for (int32_t e = 0; e < nl; ++e, o += 32) col[o] = lo_col[l0 + e], blk[o] = ~lo_idx[l0 + e];
}

// (rn(w), rn(w - rn(w))) of w = v 2^e as floats, without FP64 instructions:
// the 53-bit mantissa rounded to 24 bits (ties to even), the signed rest
// through the integer conversion, which rounds to nearest as well.  |w| <= 1;
// a w below the normal float range becomes 0, its rest below that range
// rounds to a subnormal float.
__device__ __forceinline__ float2 ff_split_rn(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ef = (int)((b >> 52) & 0x7ff), E = ef - 1023 + e;  // w in [2^E, 2^(E+1))
  if (ef == 0 || E < -126) return make_float2(0.f, 0.f);
  const unsigned sign = (unsigned)(b >> 63) << 31;
  const unsigned q = (unsigned)((b & 0xfffffffffffffLL) >> 29);  // the 23 bits below the leading one
  int rest = (int)(b & 0x1fffffff);
  const bool up = rest > (1 << 28) || (rest == (1 << 28) && (q & 1u));
  const float hi = __uint_as_float((sign | ((unsigned)(E + 127) << 23) | q) + (up ? 1u : 0u));
  if (up) rest -= 1 << 29;
  if (rest == 0) return make_float2(hi, 0.f);
  const int k = E - 52;  // lo = rest 2^k
  float lo = __int2float_rn(sign ? -rest : rest);
  const int k1 = max(k, -126), k2 = k - k1;  // two exact factors, one rounding (a subnormal result)
  lo = __fmul_rn(__fmul_rn(lo, __uint_as_float((unsigned)(max(k2, -126) + 127) << 23)),
                 __uint_as_float((unsigned)(k1 + 127) << 23));
  return make_float2(hi, lo);
}

// Values of every entry, a lane per row of the slice, 32 neighbouring rows
// writing 32 neighbouring values.
template <bool kFF>
__global__ void __launch_bounds__(256) k_slice_values(const int32_t* __restrict__ row_order, int32_t n,
                                                      const int32_t* __restrict__ ptr,
                                                      const int32_t* __restrict__ len, const int32_t* __restrict__ col,
                                                      const int32_t* __restrict__ blk, const double* __restrict__ au,
                                                      const int32_t* __restrict__ kk, float2* __restrict__ ff,
                                                      double* __restrict__ val) {
  const int32_t t = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
  if (t >= n) return;
  const int64_t p = ptr[t >> 5];
  const int lane = t & 31;
  const int32_t L = len[t];
  const int kr = kFF ? kk[row_order[t]] + 2 * kk[n] : 0;  // k_row + K (kk holds k - K)
  for (int32_t e = blockIdx.y; e < L; e += gridDim.y) {
    const int64_t o = (p + e) * 32 + lane;
    int32_t b = blk[o];
    const bool tr = b < 0;
    if (tr) b = ~b;
    const int sh = kFF ? -(kr + kk[col[o]]) : 0;
    double H[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) H[q] = au[(int64_t)b * 9 + q];
    const int64_t w = (p + e) * 288 + lane;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
      const double h = tr ? H[q % 3 * 3 + q / 3] : H[q];
      if (kFF)
        ff[w + 32 * q] = ff_split_rn(h, sh);
      else
        val[w + 32 * q] = h;
    }
  }
}

// The device has no room for the copy: none is kept (nor tried again for this row
// order), and the error of that one allocation does not stand.
static int no_room(gs_ctx ctx, gs_mat m) {
  if (cudaPeekAtLastError() != cudaErrorMemoryAllocation) return GS_ERR_CUDA;
  cudaGetLastError();
  release_sliced(ctx, m, true);
  m->sl_window = m->row_order_window;
  return GS_OK;
}

// The sliced copy with float-float (ff) or FP64 values, made on first use and
// kept with the matrix; new values (gs_fem_refill) drop the values only.
int ensure_sliced(gs_ctx ctx, gs_mat m, bool ff) {
  cudaStream_t st = ctx->stream;
  GS_TRY(ensure_row_order(ctx, m));
  const int32_t n = m->n, slices = ceil_div(n, 32);
  if (m->sl_window != m->row_order_window) {  // the row order changed
    release_sliced(ctx, m, true);
    int32_t* most = nullptr;
    void* temp = nullptr;
    const size_t tb = scan_temp_bytes(slices + 1);
    if (ctx->scratch_buf(kSlotScan, ((size_t)slices + 2) * 4, (void**)&most) != GS_OK ||
        ctx->scratch_buf(kSlotSortTemp, tb, &temp) != GS_OK ||
        ctx->alloc((void**)&m->sl_ptr, ((size_t)slices + 1) * 4) != GS_OK ||
        ctx->alloc((void**)&m->sl_len, (size_t)std::max(n, 1) * 4) != GS_OK)
      return no_room(ctx, m);
    int32_t* longest = most + slices + 1;
    GS_CUDA(cudaMemsetAsync(longest, 0, 4, st));
    { GS_PROF(ctx, GS_K_OTHER); k_slice_len<<<ceil_div(32LL * (slices + 1), 256), 256, 0, st>>>(m->row_order, m->row_ptr, m->lo_ptr, n, slices, m->sl_len, most, longest); }
    { GS_PROF(ctx, GS_K_OTHER); GS_TRY(exclusive_scan_i32(st, most, m->sl_ptr, slices + 1, temp, tb)); }
    GS_CUDA(cudaMemcpyAsync(ctx->h_pinned + 8, m->sl_ptr + slices, 4, cudaMemcpyDeviceToHost, st));
    GS_CUDA(cudaMemcpyAsync(ctx->h_pinned + 9, longest, 4, cudaMemcpyDeviceToHost, st));
    GS_CUDA(cudaStreamSynchronize(st));
    m->sl_entries = 32LL * ctx->h_pinned[8];
    m->sl_longest = ctx->h_pinned[9];
    m->sl_window = m->row_order_window;
    if (m->sl_entries > 4 * m->nnzb + (1 << 20)) return GS_OK;  // mostly padding: a row very much longer than the rest
    const size_t words = (size_t)std::max<int64_t>(m->sl_entries, 1);
    if (ctx->alloc((void**)&m->sl_blk, words * 4) != GS_OK || ctx->alloc((void**)&m->sl_col, words * 4) != GS_OK)
      return no_room(ctx, m);
    { GS_PROF(ctx, GS_K_OTHER); k_slice_entries<<<ceil_div(n, 256), 256, 0, st>>>(m->row_order, m->row_ptr, m->cid, m->lo_ptr, m->lo_idx, m->lo_col, n, m->sl_ptr, m->sl_col, m->sl_blk); }
  }
  if (!m->sl_col) return GS_OK;
  if (ff ? m->sl_ff != nullptr : m->sl_f64 != nullptr) return GS_OK;
  if (ff) {
    GS_TRY(ensure_ff_scales(ctx, m));
    if (ctx->alloc((void**)&m->sl_ff, (size_t)std::max<int64_t>(m->sl_entries, 1) * 72) != GS_OK) return no_room(ctx, m);
  } else {
    if (ctx->alloc((void**)&m->sl_f64, (size_t)std::max<int64_t>(m->sl_entries, 1) * 72) != GS_OK) return no_room(ctx, m);
  }
  GS_PROF(ctx, GS_K_OTHER);
  const dim3 grid(ceil_div(n, 256), n < 65536 ? 8 : 2);
  if (ff)
    k_slice_values<true><<<grid, 256, 0, st>>>(m->row_order, n, m->sl_ptr, m->sl_len, m->sl_col, m->sl_blk, m->au, m->ff_k, m->sl_ff, nullptr);
  else
    k_slice_values<false><<<grid, 256, 0, st>>>(m->row_order, n, m->sl_ptr, m->sl_len, m->sl_col, m->sl_blk, m->au, nullptr, nullptr, m->sl_f64);
  GS_CUDA(cudaGetLastError());
  return GS_OK;
}

// Drops the sliced values, and with `all` the structure too.
void release_sliced(gs_ctx ctx, gs_mat m, bool all) {
  ctx->release(m->sl_ff);
  ctx->release(m->sl_f64);
  m->sl_ff = nullptr;
  m->sl_f64 = nullptr;
  if (!all) return;
  ctx->release(m->sl_ptr);
  ctx->release(m->sl_len);
  ctx->release(m->sl_col);
  ctx->release(m->sl_blk);
  m->sl_ptr = m->sl_len = m->sl_col = m->sl_blk = nullptr;
  m->sl_window = -1;
}

}  // namespace gs
