// Sums of runs of 3x3 blocks, a matrix row at a time by one warp or one block (Sec.
// 5.2, the reduction of blocks with equal keys).  Shared by the assembly from
// triplets (assemble.cu) and the numeric assembly through a stored order
// (elastic.cu): both give the same bits for the same inputs.
//
// What bounds it: 72 bytes gathered and 9 FP64 additions per input, and the
// additions as much as the bytes: an FP64 instruction costs its 16 cycles per
// SM however few lanes take part (13.4M inputs: 0.19 ms of additions with full
// warps, 0.2 ms of reads).  So nine neighbouring lanes read one block (three
// blocks per warp instruction, 9 sectors), and the three lane groups take
// equal thirds of a row's entries whatever its runs are: every step is one
// addition for the whole warp.  A group per run left the warp waiting for the
// longest run (the diagonal's) at three times the additions.
// A warp alone needs 12 us for 256 entries, one batch of loads after the other, so a
// longer row is shared by the 8 or 32 warps of a block: 20,000 inputs with a row of 4,000
// assembled in 369 us by one warp, 119 so; numeric assembly of a fan of 1,000 tets (a
// row of 4,000 inputs) 287 and 102; the 40^3 body with 1,000 affine cubes, whose rows
// of bodies are 257 to 500 inputs long, 633 and 587; 1M inputs on 3,000 rows 355 and 194
// (325 with 32 warps to every row).
#pragma once

#include "primitives.cuh"

namespace gs {

constexpr int kPiece = 256;      // entries that a warp sums at a time, and the longest row of a warp alone
constexpr int kRowPiece = 128;   // entries of a longer row that one of a block's warps sums
constexpr int kMidWarps = 8, kRowMid = kMidWarps * kRowPiece;      // rows of a block of 8 warps
constexpr int kRowWarps = 32, kRowSerial = kRowWarps * kRowPiece;  // longest row of a block, summed in a fixed order

template <bool kAtomic>
__device__ __forceinline__ void put_sum(double* dst, double v) {
  if (kAtomic)
    atomicAdd(dst, v);
  else
    *dst = v;
}

// Whole warp.  Entries 0 .. m-1 (m <= kPiece, m > 0) of a row: s_idx their
// blocks, s_dst their destination blocks in R, ascending.  cv (component
// lane % 9) and cd carry the unfinished run between a row's pieces (cd = -1:
// none); the last run stays in them.  Each lane group sums its third in
// order; a run that spans groups is added group by group.  The run of destination
// `open` goes to ov instead of R (-1: none).
template <bool kAtomic>
__device__ __forceinline__ void sum_piece(const double* __restrict__ blocks, const uint32_t* s_idx,
                                          const int32_t* s_dst, int m, double* __restrict__ R, double& cv, int32_t& cd,
                                          int32_t open, double& ov, int lane) {
  constexpr int kLoads = 6;  // blocks in flight per lane group
  const int g = lane / 9, q = lane - 9 * g;
  const int T = (m + 2) / 3;
  const int b = g * T, e = g < 3 ? min(b + T, m) : b;
  const int32_t f = b < e ? s_dst[b] : -1;  // the group's first run
  int32_t cur = f;
  double acc = 0.0, lead = 0.0;
  for (int t = 0; t < T; t += kLoads) {
    double v[kLoads];
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int p = b + t + k;
      v[k] = p < e ? blocks[(size_t)s_idx[p] * 9 + q] : 0.0;
    }
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      if (t + k >= T) break;  // whole warp
      const int p = b + t + k;
      const int32_t d = p < e ? s_dst[p] : cur;
      if (d != cur) {
        if (cur == f)
          lead = acc;
        else
          put_sum<kAtomic>(R + (size_t)cur * 9 + q, acc);
        acc = 0.0;
        cur = d;
      }
      acc += v[k];
    }
  }
#pragma unroll
  for (int h = 0; h < 3; ++h) {  // the groups' first and last runs, in order
    const int from = 9 * h + lane % 9;
    const int32_t hf = __shfl_sync(kFull, f, from), hc = __shfl_sync(kFull, cur, from);
    const double first = __shfl_sync(kFull, cur == f ? acc : lead, from), last = __shfl_sync(kFull, acc, from);
    if (hf < 0) continue;  // whole warp
    if (cd >= 0 && cd != hf) {
      if (cd == open)
        ov = cv;
      else if (lane < 9)
        put_sum<kAtomic>(R + (size_t)cd * 9 + lane, cv);
    }
    cv = (cd == hf ? cv : 0.0) + first;
    cd = hf;
    if (hc != hf) {
      if (hf == open)
        ov = cv;
      else if (lane < 9)
        put_sum<kAtomic>(R + (size_t)hf * 9 + lane, cv);
      cv = last;
      cd = hc;
    }
  }
}
template <bool kAtomic>
__device__ __forceinline__ void sum_piece(const double* __restrict__ blocks, const uint32_t* s_idx,
                                          const int32_t* s_dst, int m, double* __restrict__ R, double& cv, int32_t& cd,
                                          int lane) {
  double none;
  sum_piece<kAtomic>(blocks, s_idx, s_dst, m, R, cv, cd, -1, none, lane);
}

// A row shared by the kWarps warps of a block (8 for up to kRowMid entries, else 32),
// warp w its piece w of row_piece(len) entries (fewer, or none, at the row's end).
template <int kWarps>
__device__ __forceinline__ bool row_is_mine(int len) {
  return kWarps == kMidWarps ? len <= kRowMid : len > kRowMid;
}
template <int kWarps>
__device__ __forceinline__ int row_piece(int len) {
  return (len + kWarps - 1) / kWarps;
}

// The first and last runs of the block's pieces, which may go on in the next piece.
template <int kWarps>
struct RowEnds {
  double first[kWarps][9], last[kWarps][9];
  int32_t fd[kWarps], ld[kWarps];
};

// Whole block: sums of the row's runs from each warp's piece of m entries; the pieces'
// ends are joined in order by the first warp.
template <int kWarps>
__device__ __forceinline__ void sum_row_block(const double* __restrict__ blocks, const uint32_t* s_idx,
                                              const int32_t* s_dst, int m, double* __restrict__ R, RowEnds<kWarps>* e,
                                              int w, int lane) {
  if (m > 0) {  // whole warp
    const int32_t open = s_dst[0];
    double cv = 0.0, ov = 0.0;
    int32_t cd = -1;
    sum_piece<false>(blocks, s_idx, s_dst, m, R, cv, cd, open, ov, lane);
    if (lane < 9) e->first[w][lane] = cd == open ? cv : ov, e->last[w][lane] = cv;
    if (lane == 0) e->fd[w] = open, e->ld[w] = cd;
  } else if (lane == 0) {
    e->fd[w] = -1;
  }
  __syncthreads();
  if (w > 0 || lane >= 9) return;
  double cv = 0.0;
  int32_t cd = -1;
  for (int i = 0; i < kWarps && e->fd[i] >= 0; ++i) {
    const int32_t f = e->fd[i], l = e->ld[i];
    if (cd >= 0 && cd != f) R[(size_t)cd * 9 + lane] = cv;
    cv = (cd == f ? cv : 0.0) + e->first[i][lane];
    cd = f;
    if (l != f) {
      R[(size_t)f * 9 + lane] = cv;
      cv = e->last[i][lane];
      cd = l;
    }
  }
  R[(size_t)cd * 9 + lane] = cv;
}

}  // namespace gs
