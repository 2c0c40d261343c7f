// Global Hessian assembly by hash-key reduction (Sec. 5.1-5.2).
//
// FastHashReduction: encode every consumed (row <= col) block with a key,
// radix-sort (key, input index) pairs so duplicates become adjacent, mark
// P[i] = K[i] != K[i+1], take O = ExclusiveSum(P) as each entry's unique-key
// index, and reduce runs with FastSegmentReduction (a warp head-segmented
// reduction; segments crossing a warp boundary finish with atomics).
//
// GB300 choices: the sort is a counting sort by row (one atomic per input
// counts the rows and ranks the input within its row, one scatter of 8-byte
// (column, index) keys) followed by a sort of every row's keys in a warp's
// registers or a block's shared memory; the runs of a sorted row are then
// summed by that warp or block, nine lanes to a 3x3 block (reduce_rows).  The inputs of rows of
// more than 4,096 are radix-sorted among themselves and summed by as many warps
// as they need.  Matrices of mostly empty rows take the general path: keys packed
// as (row << b) | col with b the bit width of n, which keeps the (row, col) order
// of the paper's (row << 32) | col encoding while shortening the radix sort
// to 2b bits, values gathered through the sorted index, run flags, scan and
// FastSegmentReduction (reduce_sorted_keys).
#include <cub/device/device_reduce.cuh>

#include <algorithm>

#include "common.cuh"
#include "sort_scan.cuh"
#include "primitives.cuh"
#include "run_reduce.cuh"

namespace gs {

__global__ void k_encode_keys(const int32_t* __restrict__ rows, const int32_t* __restrict__ cols, int64_t nb,
                              int32_t n, int shift, uint64_t sentinel, uint64_t* __restrict__ keys,
                              uint32_t* __restrict__ idx, int* flags) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  int32_t r = rows[i], c = cols[i];
  uint64_t key = sentinel;
  if (r < 0 || r >= n || c < 0 || c >= n) {
    atomicOr(flags, kErrIndex);
  } else if (r <= c) {
    key = ((uint64_t)r << shift) | (uint64_t)c;
  }
  keys[i] = key;
  idx[i] = (uint32_t)i;
}

// P[i] = K[i] != K[i+1]; the last entry closes the final run.
__global__ void k_run_flags(const uint64_t* __restrict__ keys, int64_t nb, int32_t* __restrict__ P) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  P[i] = (i + 1 == nb) ? 1 : (keys[i] != keys[i + 1]);
}

// FastSegmentReduction over the sorted entries.  Thread i holds the block
// of sorted entry i (gathered through idx) and its unique-key index O[i].
// The first entry of each run also writes the decoded (row, col).
__global__ void k_fast_segment_reduce(const uint64_t* __restrict__ keys, const uint32_t* __restrict__ idx,
                                      const int32_t* __restrict__ O, const double* __restrict__ blocks,
                                      int64_t nb, uint64_t sentinel, int shift, double* __restrict__ R,
                                      int32_t* __restrict__ rid, int32_t* __restrict__ cid,
                                      int32_t* __restrict__ key_of_input) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int lane = threadIdx.x & 31;
  bool in = i < nb;
  uint64_t key = in ? keys[i] : sentinel;
  bool valid = in && key != sentinel;
  int32_t b = in ? O[i] : -1;
  int32_t b_prev = (in && i > 0) ? O[i - 1] : -1;
  bool head = (lane == 0) || (b_prev != b);
  double v[9];
  if (valid) {
    const double* src = blocks + (size_t)idx[i] * 9;
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = src[k];
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) v[k] = 0.0;
  }
  unsigned hm = __ballot_sync(kFull, head);
  int send = segment_end(hm, lane);
  head_segmented_reduce<9>(v, lane, send);
  if (in) key_of_input[idx[i]] = valid ? b : -1;  // which stored block each input fed
  if (!valid) return;
  if (b_prev != b) {  // first entry of its run: record the key
    rid[b] = (int32_t)(key >> shift);
    cid[b] = (int32_t)(key & ((1ull << shift) - 1));
  }
  if (!head) return;
  // A segment that began in an earlier warp or continues into the next one
  // is shared between warps: finish it with atomics; otherwise store.
  bool cont_prev = (lane == 0) && (b_prev == b);
  bool cont_next = false;
  if (send == 32) {
    int64_t nxt = i - lane + 32;
    cont_next = nxt < nb && O[nxt] == b;
  }
  double* dst = R + (size_t)b * 9;
  if (cont_prev || cont_next) {
#pragma unroll
    for (int k = 0; k < 9; ++k) atomicAdd(dst + k, v[k]);
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) dst[k] = v[k];
  }
}

// row_ptr[r] = first stored block of row r (rows without blocks get the
// next row's start); row_ptr[n] = U.
__global__ void k_row_ptr(const int32_t* __restrict__ rid, int64_t U, int32_t n, int32_t* __restrict__ row_ptr) {
  int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u > U) return;
  int32_t r_here = (u < U) ? rid[u] : n;
  int32_t r_prev = (u > 0) ? rid[u - 1] : -1;
  for (int32_t r = r_prev + 1; r <= r_here; ++r) row_ptr[r] = (int32_t)u;
}

// ---------------------------------------------------------------- rows sorted one by one
// What bounds it: 80 bytes per input and stored block, and the additions
// (run_reduce.cuh).  A radix sort of 13.4M inputs (64^3 body) moved 24 bytes
// per key and pass, and its reduction read each 72-byte block by one thread,
// nine loads spread over 32 blocks.  Here a key is written once and read
// twice.  Measured, gs_assemble and gs_mat_export: 2.48 -> 1.25 ms (64^3, 13.4M
// inputs), 0.21 -> 0.094 ms (16^3, 0.18M), two-level 1.34 -> 0.59 ms (40^3 and
// 1,000 bodies).
constexpr int kRowWarp = kPiece;       // longest row sorted, and summed, by one warp
constexpr int kRowBlock = kRowSerial;  // longest row sorted, and summed, by one block (32 KB of keys)

// Words of the row path: rows that a block sorts, and the rows longer than
// kRowBlock as (their number << 32) | their inputs, which the host reads back.
struct RowWords {
  uint64_t huge;
  int32_t n_long, n_longer;  // of more than kRowWarp, of more than kRowMid inputs
};

// What the host waits for, and the error word (cleared), into pinned memory in one
// launch.
__global__ void k_row_words(const RowWords* __restrict__ words, const int32_t* __restrict__ total,
                            int* __restrict__ flags, int* __restrict__ host) {
  host[0] = *flags;
  *flags = 0;
  host[4] = (int)(words->huge >> 32);
  host[5] = (int)(uint32_t)words->huge;
  host[6] = words->n_long;
  host[7] = words->n_longer;
  host[8] = *total;
}

// Whole warp: each counting lane's rank in its row's count cnt[r], in no fixed order.
// The lanes of the warp's first four rows add once per row: a row of very many inputs
// (the reduced rows of a body of thousands of nodes) is one address for all of them,
// and 2M atomics on four addresses took 0.7 ms, 0.19 so.
__device__ __forceinline__ int32_t rank_in_row(int32_t* cnt, int32_t r, bool counts, int lane) {
  uint32_t left = __ballot_sync(kFull, counts), group = 1u << lane;  // lanes that add with this one
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (!left) break;  // whole warp
    const int32_t rl = __shfl_sync(kFull, r, __ffs(left) - 1);
    const bool mine = counts && r == rl;
    const uint32_t same = __ballot_sync(kFull, mine);
    if (mine) group = same;
    left &= ~same;
  }
  const int lead = __ffs(group) - 1;
  int32_t first = 0;
  if (counts && lane == lead) first = atomicAdd(&cnt[r], __popc(group));
  first = __shfl_sync(kFull, first, lead);
  return counts ? first + __popc(group & ((1u << lane) - 1u)) : -1;
}

// An input that counts is inside and on or above the diagonal.
__device__ __forceinline__ bool input_counts(int32_t r, int32_t c, int32_t n, int* flags) {
  if (r < 0 || r >= n || c < 0 || c >= n) {
    atomicOr(flags, kErrIndex);
    return false;
  }
  return r <= c;
}

// Counts the rows' inputs and ranks each within its row.
__global__ void k_row_count(const int32_t* __restrict__ rows, const int32_t* __restrict__ cols, int64_t nb, int32_t n,
                            int32_t* __restrict__ cnt, int32_t* __restrict__ rank, int32_t* __restrict__ key_of_input,
                            int* __restrict__ flags) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = i < nb;
  const int32_t r = in ? rows[i] : 0;
  const bool counts = in && input_counts(r, cols[i], n, flags);
  const int32_t k = rank_in_row(cnt, r, counts, threadIdx.x & 31);
  if (!in) return;
  rank[i] = k;
  if (!counts) key_of_input[i] = -1;
}

// The same where few rows take many inputs each: their counts lie in a few lines, whose
// atomics one slice of the L2 serves (1M inputs on 300 rows: 197 us).  A block ranks
// its chunk of inputs against counts in shared memory and adds those to the rows' once
// (11 us).
constexpr int32_t kFewRows = 8192;      // counts of 32 KB
constexpr int kFewInputs = 256;         // inputs per row and more
__global__ void __launch_bounds__(1024) k_row_count_few(const int32_t* __restrict__ rows,
                                                        const int32_t* __restrict__ cols, int64_t nb, int32_t n,
                                                        int64_t chunk, int32_t* __restrict__ cnt,
                                                        int32_t* __restrict__ rank, int32_t* __restrict__ key_of_input,
                                                        int* __restrict__ flags) {
  extern __shared__ int32_t s_cnt[];  // the chunk's counts, then where they begin in the rows'
  const int lane = threadIdx.x & 31;
  const int64_t i0 = blockIdx.x * chunk, i1 = min(i0 + chunk, nb);
  for (int r = threadIdx.x; r < n; r += blockDim.x) s_cnt[r] = 0;
  __syncthreads();
  for (int64_t j = i0; j < i1; j += blockDim.x) {  // whole block
    const int64_t i = j + threadIdx.x;
    const bool in = i < i1;
    const int32_t r = in ? rows[i] : 0;
    const bool counts = in && input_counts(r, cols[i], n, flags);
    const int32_t k = rank_in_row(s_cnt, r, counts, lane);
    if (in) {
      rank[i] = k;
      if (!counts) key_of_input[i] = -1;
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x)
    if (s_cnt[r]) s_cnt[r] = atomicAdd(&cnt[r], s_cnt[r]);
  __syncthreads();
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x)  // this thread's own ranks
    if (rank[i] >= 0) rank[i] += s_cnt[rows[i]];
}

// The ranks of a row's inputs are in no fixed order; the sort by (column,
// input index) that follows makes it one.
__global__ void k_row_scatter(const int32_t* __restrict__ rows, const int32_t* __restrict__ cols,
                              const int32_t* __restrict__ rank, const int32_t* __restrict__ start, int64_t nb,
                              uint64_t* __restrict__ list) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  const int32_t k = rank[i];
  if (k >= 0) list[(int64_t)start[rows[i]] + k] = ((uint64_t)(uint32_t)cols[i] << 32) | (uint32_t)i;
}

// Bitonic sort of 32 kR keys, element q * 32 + lane in a[q]; then the sorted
// keys go back and the distinct columns are counted.
template <int kR>
__device__ __forceinline__ int32_t sort_row(uint64_t* __restrict__ row, int32_t len, int lane) {
  uint64_t a[kR];
#pragma unroll
  for (int q = 0; q < kR; ++q) a[q] = q * 32 + lane < len ? row[q * 32 + lane] : ~0ull;
#pragma unroll
  for (int k = 2; k <= 32 * kR; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
#pragma unroll
        for (int q = 0; q < kR; ++q) {
          const int o = q ^ (j / 32);
          if (o > q) {
            const bool up = ((q * 32) & k) == 0;
            const uint64_t lo = a[q] < a[o] ? a[q] : a[o], hi = a[q] < a[o] ? a[o] : a[q];
            a[q] = up ? lo : hi, a[o] = up ? hi : lo;
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < kR; ++q) {
          const uint64_t b = __shfl_xor_sync(kFull, a[q], j);
          const bool up = (k < 32 ? (lane & k) : ((q * 32) & k)) == 0;
          const bool keep_min = up == ((lane & j) == 0);
          a[q] = (a[q] < b) == keep_min ? a[q] : b;
        }
      }
    }
  }
  int32_t unique = 0;
#pragma unroll
  for (int q = 0; q < kR; ++q) {
    const uint32_t c = (uint32_t)(a[q] >> 32);
    uint32_t p = __shfl_up_sync(kFull, c, 1);
    if (q > 0) {
      const uint32_t last = __shfl_sync(kFull, (uint32_t)(a[q - 1] >> 32), 31);
      if (lane == 0) p = last;
    }
    const bool in = q * 32 + lane < len;
    if (in) row[q * 32 + lane] = a[q];
    unique += __popc(__ballot_sync(kFull, in && (c != p || (q == 0 && lane == 0))));
  }
  return unique;
}

// Rows of up to kRowWarp inputs; the others go to the lists of k_row_sort_block
// (long_rows, from the front) and of the huge rows (long_rows, from the back, and
// their first places among all inputs of huge rows).
__global__ void __launch_bounds__(256) k_row_sort(const int32_t* __restrict__ start, int32_t n,
                                                  uint64_t* __restrict__ list, int32_t* __restrict__ unique,
                                                  RowWords* __restrict__ words, int32_t* __restrict__ long_rows,
                                                  int32_t* __restrict__ huge_base) {
  const int32_t r = (int32_t)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= n) return;  // whole warp
  const int32_t s0 = start[r], len = start[r + 1] - s0;
  uint64_t* row = list + s0;
  int32_t u = 0;
  if (len > kRowWarp) {
    if (lane == 0) {
      if (len > kRowBlock) {
        const uint64_t old =
            atomicAdd((unsigned long long*)&words->huge, (1ull << 32) | (unsigned long long)(uint32_t)len);
        const int32_t h = (int32_t)(old >> 32);
        long_rows[n - 1 - h] = r;
        huge_base[h] = (int32_t)(uint32_t)old;
      } else {
        long_rows[atomicAdd(&words->n_long, 1)] = r;
        if (len > kRowMid) atomicAdd(&words->n_longer, 1);
      }
    }
    return;  // k_row_sort_block or k_huge_unique writes this row's count
  }
  if (len > 128)
    u = sort_row<8>(row, len, lane);
  else if (len > 64)
    u = sort_row<4>(row, len, lane);
  else if (len > 32)
    u = sort_row<2>(row, len, lane);
  else if (len > 0)
    u = sort_row<1>(row, len, lane);
  if (lane == 0) unique[r] = u;
}

// The long rows, a block each.
constexpr int kSortBlock = 512;  // threads of it
__global__ void __launch_bounds__(kSortBlock) k_row_sort_block(const int32_t* __restrict__ start, uint64_t* __restrict__ list,
                                                        int32_t* __restrict__ unique,
                                                        const RowWords* __restrict__ words,
                                                        const int32_t* __restrict__ long_rows) {
  __shared__ uint64_t a[kRowBlock];
  __shared__ int32_t s_unique;
  const int32_t n_long = words->n_long;
  for (int32_t w = blockIdx.x; w < n_long; w += gridDim.x) {
    const int32_t r = long_rows[w], s0 = start[r], len = start[r + 1] - s0;
    int size = 2 * kRowWarp;
    while (size < len) size *= 2;
    for (int e = threadIdx.x; e < size; e += blockDim.x) a[e] = e < len ? list[s0 + e] : ~0ull;
    if (threadIdx.x == 0) s_unique = 0;
    __syncthreads();
    for (int k = 2; k <= size; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = threadIdx.x; t < size / 2; t += blockDim.x) {
          const int e = 2 * t - (t & (j - 1)), o = e + j;  // the pairs that differ in bit j
          const uint64_t x = a[e], y = a[o];
          if ((x > y) == ((e & k) == 0)) a[e] = y, a[o] = x;
        }
        __syncthreads();
      }
    int32_t u = 0;
    for (int e = threadIdx.x; e < len; e += blockDim.x) {
      list[s0 + e] = a[e];
      u += e == 0 || (a[e] >> 32) != (a[e - 1] >> 32);
    }
    atomicAdd(&s_unique, u);
    __syncthreads();
    if (threadIdx.x == 0) unique[r] = s_unique;
    __syncthreads();
  }
}

// Keys of a piece of m sorted entries from entry p0 of row r (list: the row's), whose
// first run is the stored block `next` where it begins with a head, else next - 1:
// each input's stored block, and the runs' keys.
__device__ __forceinline__ void number_runs(const uint64_t* __restrict__ list, int32_t p0, int m, int32_t r,
                                            int32_t next, uint32_t* s_idx, int32_t* s_dst, int32_t* __restrict__ rid,
                                            int32_t* __restrict__ cid, int32_t* __restrict__ key_of_input, int lane) {
  uint32_t before = p0 > 0 ? (uint32_t)(list[p0 - 1] >> 32) : 0;  // column of the entry ahead
  for (int j = 0; j < m; j += 32) {
    const int32_t p = p0 + j + lane;
    const bool in = j + lane < m;
    const uint64_t key = in ? list[p] : ~0ull;
    const uint32_t c = (uint32_t)(key >> 32);
    uint32_t prev = __shfl_up_sync(kFull, c, 1);
    if (lane == 0) prev = before;
    before = __shfl_sync(kFull, c, 31);
    const bool head = in && (p == 0 || c != prev);
    const uint32_t hm = __ballot_sync(kFull, head);
    const int32_t u = next + __popc(hm & (0xffffffffu >> (31 - lane))) - 1;
    if (head) {
      rid[u] = r;
      cid[u] = (int32_t)c;
    }
    if (in) {
      s_idx[j + lane] = (uint32_t)key;
      s_dst[j + lane] = u;
      key_of_input[(uint32_t)key] = u;
    }
    next += __popc(hm);
  }
}

// The runs of every sorted row of up to kPiece inputs, a warp per row: finds the runs,
// writes their keys and each input's stored block, and sums them (run_reduce.cuh).
__global__ void __launch_bounds__(256) k_row_reduce(const int32_t* __restrict__ start,
                                                    const int32_t* __restrict__ row_ptr,
                                                    const uint64_t* __restrict__ list,
                                                    const double* __restrict__ blocks, int32_t n,
                                                    double* __restrict__ R, int32_t* __restrict__ rid,
                                                    int32_t* __restrict__ cid, int32_t* __restrict__ key_of_input) {
  __shared__ uint32_t s_idx[8][kPiece];
  __shared__ int32_t s_dst[8][kPiece];
  const int32_t r = (int32_t)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (r >= n) return;  // whole warp
  const int32_t s0 = start[r], len = start[r + 1] - s0;
  if (len == 0 || len > kPiece) return;
  number_runs(list + s0, 0, len, r, row_ptr[r], s_idx[w], s_dst[w], rid, cid, key_of_input, lane);
  __syncwarp();
  double cv = 0.0;
  int32_t cd = -1;
  sum_piece<false>(blocks, s_idx[w], s_dst[w], len, R, cv, cd, lane);
  if (lane < 9) R[(size_t)cd * 9 + lane] = cv;
}

// The same for the rows that a block sorted, a block each; those of the other kWarps
// return.
template <int kWarps>
__global__ void __launch_bounds__(32 * kWarps) k_row_reduce_block(
    const int32_t* __restrict__ start, const int32_t* __restrict__ row_ptr, const uint64_t* __restrict__ list,
    const double* __restrict__ blocks, const int32_t* __restrict__ long_rows, double* __restrict__ R,
    int32_t* __restrict__ rid, int32_t* __restrict__ cid, int32_t* __restrict__ key_of_input) {
  __shared__ uint32_t s_idx[kWarps][kRowPiece];
  __shared__ int32_t s_dst[kWarps][kRowPiece];
  __shared__ RowEnds<kWarps> ends;
  __shared__ int s_heads[kWarps];
  const int32_t r = long_rows[blockIdx.x];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int32_t s0 = start[r], len = start[r + 1] - s0;
  if (!row_is_mine<kWarps>(len)) return;  // whole block
  const int per = row_piece<kWarps>(len), p0 = w * per, m = max(0, min(per, len - p0));
  const uint64_t* row = list + s0;
  int heads = 0;
  for (int j = lane; j < m; j += 32) {
    const int32_t p = p0 + j;
    heads += p == 0 || (row[p] >> 32) != (row[p - 1] >> 32);
  }
  heads = __reduce_add_sync(kFull, heads);
  if (lane == 0) s_heads[w] = heads;
  __syncthreads();
  int32_t next = row_ptr[r];
  for (int i = 0; i < w; ++i) next += s_heads[i];
  if (m > 0) number_runs(row, p0, m, r, next, s_idx[w], s_dst[w], rid, cid, key_of_input, lane);  // whole warp
  __syncwarp();
  sum_row_block<kWarps>(blocks, s_idx[w], s_dst[w], m, R, &ends, w, lane);
}

// ---------------------------------------------------------------- rows of more than kRowBlock inputs
// Their inputs are sorted together by (row's number h, column) in one radix
// sort, and summed in pieces of 256 sorted entries (64 where 256 would leave SMs
// idle) whatever the rows are, a warp each, added to the zeroed output.  The other
// rows are summed as ever.  Sending the whole matrix to the general path instead,
// once the row path had met a row too long for it, paid for both: 13.4M inputs with
// one row of 5,000 2.72 ms (0.81 so; 2.25 in the general path alone), 2M inputs on
// four rows 1.48 (0.57; 0.78), a two-level assembly with a body of 8,192 nodes 0.99
// (0.45; 0.85), 20,000 inputs with a row of 4,200 0.165 (0.126; 0.149).  The inputs of
// one block are summed in no fixed order here (as a run of several pieces is anyway):
// the input's number as a third part of the key cost two or three more passes.
__global__ void k_huge_keys(const uint64_t* __restrict__ list, const int32_t* __restrict__ start,
                            const int32_t* __restrict__ last_row, const int32_t* __restrict__ base, int32_t n_huge,
                            int32_t m, int cb, uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= m) return;
  int32_t lo = 0, hi = n_huge;  // base[lo] <= p < base[hi]
  while (hi - lo > 1) {
    const int32_t mid = (lo + hi) / 2;
    if (base[mid] <= p)
      lo = mid;
    else
      hi = mid;
  }
  const uint64_t e = list[(int64_t)start[*(last_row - lo)] + (p - base[lo])];
  keys[p] = ((uint64_t)lo << cb) | (e >> 32);
  vals[p] = (uint32_t)e;
}

// head[p]: sorted entry p begins a run (head[m]: 0, the end of the scan).
__global__ void k_huge_heads(const uint64_t* __restrict__ keys, int32_t m, int32_t* __restrict__ head) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p <= m) head[p] = p < m && (p == 0 || keys[p] != keys[p - 1]);
}

__global__ void k_huge_unique(const int32_t* __restrict__ last_row, const int32_t* __restrict__ base, int32_t n_huge,
                              int32_t m, const int32_t* __restrict__ before, int32_t* __restrict__ unique) {
  const int32_t h = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x);
  if (h < n_huge) unique[*(last_row - h)] = before[h + 1 < n_huge ? base[h + 1] : m] - before[base[h]];
}

__global__ void __launch_bounds__(256) k_huge_reduce(const uint64_t* __restrict__ keys,
                                                     const uint32_t* __restrict__ vals,
                                                     const int32_t* __restrict__ before,
                                                     const int32_t* __restrict__ last_row,
                                                     const int32_t* __restrict__ base, int32_t m, int piece, int cb,
                                                     const int32_t* __restrict__ row_ptr,
                                                     const double* __restrict__ blocks, double* __restrict__ R,
                                                     int32_t* __restrict__ rid, int32_t* __restrict__ cid,
                                                     int32_t* __restrict__ key_of_input) {
  __shared__ uint32_t s_idx[8][kPiece];
  __shared__ int32_t s_dst[8][kPiece];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t p0 = ((int64_t)blockIdx.x * 8 + w) * piece;
  if (p0 >= m) return;  // whole warp
  const int len = (int)min((int64_t)piece, m - p0);
  for (int j = lane; j < len; j += 32) {
    const int64_t p = p0 + j;
    const uint64_t key = keys[p];
    const int32_t h = (int32_t)(key >> cb), r = *(last_row - h);
    const int32_t u = row_ptr[r] + before[p + 1] - 1 - before[base[h]];
    const uint32_t i = vals[p];
    if (before[p + 1] != before[p]) {
      rid[u] = r;
      cid[u] = (int32_t)(key & ((1ull << cb) - 1));
    }
    s_idx[w][j] = i;
    s_dst[w][j] = u;
    key_of_input[i] = u;
  }
  __syncwarp();
  double cv = 0.0;
  int32_t cd = -1;
  sum_piece<true>(blocks, s_idx[w], s_dst[w], len, R, cv, cd, lane);
  if (lane < 9) atomicAdd(R + (size_t)cd * 9 + lane, cv);
}

// Sorted entries of the rows of more than kRowBlock inputs.
struct HugeRows {
  const int32_t *last_row, *base;  // row h at last_row[-h]; its first place
  int32_t n, m;                    // rows, inputs
  int cb;                          // bits of a column
  uint64_t* keys;
  uint32_t* vals;
  int32_t* before;  // runs before a sorted entry (m + 1)
};

// Sorts the huge rows' inputs and writes their unique counts.  rank's slot takes
// the sort's values.
static int sort_huge_rows(gs_ctx ctx, const uint64_t* list, const int32_t* start, int64_t nb, int32_t* unique,
                          HugeRows& g) {
  cudaStream_t st = ctx->stream;
  const int T = 256;
  uint64_t* keys = nullptr;
  uint32_t* vals = nullptr;
  void* temp = nullptr;
  const size_t tb = std::max(radix_sort_temp_bytes(g.m), scan_temp_bytes((int64_t)g.m + 1));
  GS_TRY(ctx->scratch_buf(kSlotSortKeysOut, (size_t)g.m * 16, (void**)&keys));
  GS_TRY(ctx->scratch_buf(kSlotSortValsIn, (size_t)nb * 4, (void**)&vals));
  GS_TRY(ctx->scratch_buf(kSlotSortValsOut, (size_t)g.m * 4, (void**)&g.vals));
  GS_TRY(ctx->scratch_buf(kSlotSortTemp, tb, &temp));
  g.keys = keys + g.m;
  g.before = (int32_t*)keys;  // the unsorted keys' place
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_huge_keys<<<ceil_div(g.m, T), T, 0, st>>>(list, start, g.last_row, g.base, g.n, g.m, g.cb, keys, vals); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(radix_sort_pairs(st, keys, g.keys, vals, g.vals, g.m, bits_for(g.n) + g.cb, temp, tb)); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_huge_heads<<<ceil_div((int64_t)g.m + 1, T), T, 0, st>>>(g.keys, g.m, g.before); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(exclusive_scan_i32(st, g.before, g.before, (int64_t)g.m + 1, temp, tb)); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_huge_unique<<<ceil_div(g.n, T), T, 0, st>>>(g.last_row, g.base, g.n, g.m, g.before, unique); }
  return GS_OK;
}

// Rows sorted one by one.
static int reduce_rows(gs_ctx ctx, gs_mat m, const int32_t* rows, const int32_t* cols, const double* blocks,
                       int64_t nb) {
  cudaStream_t st = ctx->stream;
  const int32_t n = m->n;
  const int T = 256;
  // counts / unique counts, row starts, worklists of long and huge rows, words
  int32_t* rank = nullptr;
  uint64_t* list = nullptr;
  void* temp = nullptr;
  const size_t tb = scan_temp_bytes((int64_t)n + 1);
  RowWords* words = nullptr;  // then the counts
  const size_t ints = 3 * (size_t)n + 2 + (size_t)(nb / kRowBlock) + 1;
  GS_TRY(ctx->scratch_buf(kSlotScan, sizeof(RowWords) + ints * 4, (void**)&words));
  GS_TRY(ctx->scratch_buf(kSlotSortValsIn, (size_t)nb * 4, (void**)&rank));
  GS_TRY(ctx->scratch_buf(kSlotSortKeysIn, (size_t)nb * 8, (void**)&list));
  GS_TRY(ctx->scratch_buf(kSlotSortTemp, tb, &temp));
  int32_t *cnt = (int32_t*)(words + 1), *start = cnt + n + 1, *long_rows = start + n + 1, *huge_base = long_rows + n;
  GS_CUDA(cudaMemsetAsync(words, 0, sizeof(RowWords) + ((size_t)n + 1) * 4, st));
  if (n <= kFewRows && nb >= (int64_t)kFewInputs * n && nb >= 16384) {
    // eight inputs and more per row and chunk, four inputs and more per thread
    const int64_t chunk = std::max<int64_t>(4096, (8LL * n + 1023) / 1024 * 1024);
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_row_count_few<<<ceil_div(nb, chunk), 1024, (size_t)n * 4, st>>>(rows, cols, nb, n, chunk, cnt, rank, m->key_of_input, ctx->d_flags);
  } else {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_row_count<<<ceil_div(nb, T), T, 0, st>>>(rows, cols, nb, n, cnt, rank, m->key_of_input, ctx->d_flags);
  }
  { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(exclusive_scan_i32(st, cnt, start, (int64_t)n + 1, temp, tb)); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_row_scatter<<<ceil_div(nb, T), T, 0, st>>>(rows, cols, rank, start, nb, list); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_row_sort<<<ceil_div(32LL * n, T), T, 0, st>>>(start, n, list, cnt, words, long_rows, huge_base); }
  {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_row_sort_block<<<std::max(1, std::min(4 * ctx->sm_count, n)), kSortBlock, 0, st>>>(start, list, cnt, words, long_rows);
  }
  HugeRows huge{};
  for (int pass = 0;; ++pass) {
    { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(exclusive_scan_i32(st, cnt, m->row_ptr, (int64_t)n + 1, temp, tb)); }
    k_row_words<<<1, 1, 0, st>>>(words, m->row_ptr + n, ctx->d_flags, ctx->h_pinned);
    GS_CUDA(cudaGetLastError());
    GS_TRY(ctx->sync());
    if (ctx->h_pinned[0]) return status_from_flags(ctx->h_pinned[0]);
    huge.n = ctx->h_pinned[4], huge.m = ctx->h_pinned[5];
    if (pass || !huge.n) break;
    huge.last_row = long_rows + n - 1, huge.base = huge_base;
    huge.cb = bits_for(n);
    GS_TRY(sort_huge_rows(ctx, list, start, nb, cnt, huge));
    GS_TRY(ctx->scratch_buf(kSlotSortTemp, tb, &temp));  // may have grown
  }
  const int64_t U = ctx->h_pinned[8];
  m->nnzb = U;
  GS_TRY(ctx->alloc((void**)&m->au, (size_t)U * 72));
  GS_TRY(ctx->alloc((void**)&m->rid, (size_t)U * 4));
  GS_TRY(ctx->alloc((void**)&m->cid, (size_t)U * 4));
  if (U > 0) {
    if (huge.n) GS_CUDA(cudaMemsetAsync(m->au, 0, (size_t)U * 72, st));
    { GS_PROF(ctx, GS_K_ASSEMBLE); k_row_reduce<<<ceil_div(32LL * n, T), T, 0, st>>>(start, m->row_ptr, list, blocks, n, m->au, m->rid, m->cid,
                                                                                    m->key_of_input); }
  }
  const int n_long = ctx->h_pinned[6], n_longer = ctx->h_pinned[7];
  if (n_long > n_longer) {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_row_reduce_block<kMidWarps><<<n_long, 32 * kMidWarps, 0, st>>>(start, m->row_ptr, list, blocks, long_rows, m->au, m->rid, m->cid, m->key_of_input);
  }
  if (n_longer) {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_row_reduce_block<kRowWarps><<<n_long, 32 * kRowWarps, 0, st>>>(start, m->row_ptr, list, blocks, long_rows, m->au, m->rid, m->cid, m->key_of_input);
  }
  if (huge.n) {
    GS_PROF(ctx, GS_K_ASSEMBLE);
    const int piece = huge.m <= 2 * 8 * 64 * std::max(ctx->sm_count, 1) ? 64 : kPiece;  // 2 blocks per SM
    k_huge_reduce<<<ceil_div(huge.m, 8 * piece), T, 0, st>>>(huge.keys, huge.vals, huge.before, huge.last_row, huge.base, huge.m, piece,
                                                             huge.cb, m->row_ptr, blocks, m->au, m->rid, m->cid, m->key_of_input);
  }
  return GS_OK;
}

// The general path: radix sort of (key, input) pairs, run flags, exclusive
// scan, FastSegmentReduction.
static int reduce_sorted_keys(gs_ctx ctx, gs_mat m, const int32_t* rows, const int32_t* cols, const double* blocks,
                              int64_t nb) {
  cudaStream_t st = ctx->stream;
  const int32_t n = m->n;
  const int shift = bits_for(n);
  const uint64_t sentinel = (shift * 2 >= 64) ? ~0ull : ((1ull << (2 * shift)) - 1);
  const int end_bit = 2 * shift;
  uint64_t *k_in = nullptr, *k_out = nullptr;
  uint32_t *i_in = nullptr, *i_out = nullptr;
  int32_t *P = nullptr, *O = nullptr;
  const int T = 256;
  GS_TRY(ctx->scratch_buf(kSlotSortKeysIn, nb * 8, (void**)&k_in));
  GS_TRY(ctx->scratch_buf(kSlotSortKeysOut, nb * 8, (void**)&k_out));
  GS_TRY(ctx->scratch_buf(kSlotSortValsIn, nb * 4, (void**)&i_in));
  GS_TRY(ctx->scratch_buf(kSlotSortValsOut, nb * 4, (void**)&i_out));
  GS_TRY(ctx->scratch_buf(kSlotScan, nb * 8, (void**)&P));
  O = P + nb;
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_encode_keys<<<ceil_div(nb, T), T, 0, st>>>(rows, cols, nb, n, shift, sentinel, k_in, i_in, ctx->d_flags); }
  // radix sort of (key, index) and the exclusive scan of the run flags
  // (sort_scan.cu: hand-written, stable)
  const size_t tb = std::max(radix_sort_temp_bytes(nb), scan_temp_bytes(nb));
  void* temp = nullptr;
  GS_TRY(ctx->scratch_buf(kSlotSortTemp, tb, &temp));
  { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(radix_sort_pairs(st, k_in, k_out, i_in, i_out, nb, end_bit, temp, tb)); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_run_flags<<<ceil_div(nb, T), T, 0, st>>>(k_out, nb, P); }
  { GS_PROF(ctx, GS_K_ASSEMBLE); GS_TRY(exclusive_scan_i32(st, P, O, nb, temp, tb)); }
  // U = distinct keys, minus the sentinel group if present.
  uint64_t* hk = (uint64_t*)(ctx->h_pinned + 4);
  int32_t* ho = (int32_t*)(ctx->h_pinned + 8);
  GS_CUDA(cudaMemcpyAsync(hk, k_out + nb - 1, 8, cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaMemcpyAsync(ho, O + nb - 1, 4, cudaMemcpyDeviceToHost, st));
  int flags = 0;
  GS_TRY(ctx->take_flags(&flags));
  if (flags) return status_from_flags(flags);
  const int64_t U = (int64_t)ho[0] + 1 - (hk[0] == sentinel ? 1 : 0);
  m->nnzb = U;
  GS_TRY(ctx->alloc((void**)&m->au, (size_t)U * 72));
  GS_TRY(ctx->alloc((void**)&m->rid, (size_t)U * 4));
  GS_TRY(ctx->alloc((void**)&m->cid, (size_t)U * 4));
  if (U > 0) {
    GS_CUDA(cudaMemsetAsync(m->au, 0, (size_t)U * 72, st));
    GS_PROF(ctx, GS_K_ASSEMBLE);
    k_fast_segment_reduce<<<ceil_div(nb, T), T, 0, st>>>(k_out, i_out, O, blocks, nb, sentinel, shift, m->au, m->rid,
                                                         m->cid, m->key_of_input);
  } else {
    GS_CUDA(cudaMemsetAsync(m->key_of_input, 0xff, (size_t)nb * 4, st));
  }
  { GS_PROF(ctx, GS_K_ASSEMBLE); k_row_ptr<<<ceil_div(U + 1, 256), 256, 0, st>>>(m->rid, U, n, m->row_ptr); }
  return GS_OK;
}

// Reduce (rows, cols, blocks) to a new matrix.  Shared by gs_assemble and
// the second level of gs_assemble_abd.
int reduce_blocks(gs_ctx ctx, int32_t n, const int32_t* rows, const int32_t* cols, const double* blocks,
                  int64_t nb, gs_mat* out) {
  gs_mat m = new gs_mat_s();
  m->n = n;
  m->owner = ctx;
  m->n_input = nb;
  auto run = [&]() -> int {
    GS_TRY(ctx->alloc((void**)&m->key_of_input, (size_t)std::max<int64_t>(nb, 1) * 4));
    GS_TRY(ctx->alloc((void**)&m->row_ptr, (size_t)(n + 1) * 4));
    if (nb == 0) {
      int flags = 0;
      GS_TRY(ctx->take_flags(&flags));
      if (flags) return status_from_flags(flags);
      GS_CUDA(cudaMemsetAsync(m->row_ptr, 0, (size_t)(n + 1) * 4, ctx->stream));
      return GS_OK;
    }
    // Every row, empty ones too, costs the row path a warp twice, 0.44 ns, an input 0.08;
    // the general path 0.2 to 0.3 an input and a few launches more: the row path up to
    // 400,000 rows (200,000 inputs 0.22 / 0.25 ms) and where a row has three inputs
    // (1M rows: 2M inputs 0.70 / 0.60, 4M 0.84 / 0.98; 2M rows: 4M 1.36 / 1.04, 8M 1.64 /
    // 1.95).  And where few rows are so long that all would be sorted together, the
    // general path's passes are no more (50 rows, 200,000 inputs 0.24 / 0.15; 4 rows 0.20 /
    // 0.14, 1M inputs 0.31 / 0.35).
    const bool together = (n < 256 && nb >= 2304LL * n && (n > 8 || nb < 400000)) || (n < 1024 && n > 8 && nb >= 4096LL * n);
    if ((n <= 400000 || 3LL * n <= nb) && !together)
      GS_TRY(reduce_rows(ctx, m, rows, cols, blocks, nb));
    else
      GS_TRY(reduce_sorted_keys(ctx, m, rows, cols, blocks, nb));
    GS_CUDA(cudaGetLastError());
    return GS_OK;
  };
  const int s = run();
  if (s != GS_OK) {
    gs_mat_destroy(m);
    return s;
  }
  *out = m;
  return GS_OK;
}

}  // namespace gs

using namespace gs;

extern "C" {

int gs_assemble(gs_ctx ctx, int32_t n, const int32_t* rows, const int32_t* cols, const double* blocks,
                int64_t nb, gs_mat* out) {
  GS_CHECK(ctx && out, GS_ERR_INVALID, "gs_assemble: null context or output");
  *out = nullptr;
  GS_CHECK(n > 0 && n < (1 << 30), GS_ERR_INVALID, "gs_assemble: n_block_rows %d out of range", n);
  GS_CHECK(nb >= 0 && nb < (1LL << 31), GS_ERR_INVALID, "gs_assemble: n_blocks %lld out of range", (long long)nb);
  GS_CHECK(nb == 0 || (rows && cols && blocks), GS_ERR_INVALID, "gs_assemble: null input");
  GS_CUDA(cudaSetDevice(ctx->device));
  return reduce_blocks(ctx, n, rows, cols, blocks, nb, out);
}

int gs_mat_info(gs_mat m, int32_t* n, int64_t* nnzb) {
  GS_CHECK(m, GS_ERR_INVALID, "gs_mat_info: null matrix");
  if (n) *n = m->n;
  if (nnzb) *nnzb = m->nnzb;
  return GS_OK;
}

int gs_mat_export(gs_ctx ctx, gs_mat m, int32_t* rid, int32_t* cid, double* au) {
  GS_CHECK(ctx && m, GS_ERR_INVALID, "gs_mat_export: null argument");
  cudaStream_t st = ctx->stream;
  if (m->nnzb == 0) return GS_OK;
  if (rid) GS_CUDA(cudaMemcpyAsync(rid, m->rid, m->nnzb * 4, cudaMemcpyDeviceToDevice, st));
  if (cid) GS_CUDA(cudaMemcpyAsync(cid, m->cid, m->nnzb * 4, cudaMemcpyDeviceToDevice, st));
  if (au) GS_CUDA(cudaMemcpyAsync(au, m->au, m->nnzb * 72, cudaMemcpyDeviceToDevice, st));
  return GS_OK;
}

int gs_mat_destroy(gs_mat m) {
  if (!m) return GS_OK;
  gs_ctx c = m->owner;
  c->release(m->au);
  c->release(m->rid);
  c->release(m->cid);
  c->release(m->row_ptr);
  c->release(m->lo_ptr);
  c->release(m->lo_idx);
  c->release(m->lo_col);
  c->release(m->au32);
  c->release(m->au_ff);
  c->release(m->ff_k);
  c->release(m->row_order);
  gs::release_sliced(c, m, true);
  c->release(m->key_of_input);
  delete m;
  return GS_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ measurement
// Segmented reduction of already sorted keys, for comparing the paper's
// FastHashReduction (run flags + exclusive scan + warp head-segmented
// reduction, Sec. 5.2) with a library reduce-by-key on the same input.
namespace gs {
struct Block9 {
  double v[9];
};
struct Sum9 {
  __device__ __forceinline__ Block9 operator()(const Block9& a, const Block9& b) const {
    Block9 c;
#pragma unroll
    for (int k = 0; k < 9; ++k) c.v[k] = a.v[k] + b.v[k];
    return c;
  }
};
__global__ void k_iota(uint32_t* __restrict__ a, int64_t n) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = (uint32_t)i;
}
}  // namespace gs

extern "C" int gs_micro_segment_reduce(gs_ctx ctx, int64_t nb, const uint64_t* keys, const double* blocks,
                                       int32_t method, double* out, int64_t* n_unique, float* ms) {
  using namespace gs;
  GS_CHECK(ctx && keys && blocks && out && n_unique && ms && nb > 0 && nb < (1LL << 31), GS_ERR_INVALID,
           "gs_micro_segment_reduce: bad argument");
  GS_CHECK(method == 0 || method == 1, GS_ERR_INVALID, "gs_micro_segment_reduce: method %d", method);
  GS_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  cudaEvent_t e0, e1;
  GS_CUDA(cudaEventCreate(&e0));
  GS_CUDA(cudaEventCreate(&e1));
  int s = GS_OK;
  void* temp = nullptr;
  size_t tb = 0;
  int32_t *P = nullptr, *rid = nullptr, *cid = nullptr, *koi = nullptr;
  uint32_t* idx = nullptr;
  uint64_t* ukeys = nullptr;
  int64_t* nruns = nullptr;
  const int T = 256;
  if (method == 0) {
    if ((s = ctx->alloc((void**)&P, (size_t)nb * 8)) || (s = ctx->alloc((void**)&idx, (size_t)nb * 4)) ||
        (s = ctx->alloc((void**)&rid, (size_t)nb * 4)) || (s = ctx->alloc((void**)&cid, (size_t)nb * 4)) ||
        (s = ctx->alloc((void**)&koi, (size_t)nb * 4)))
      goto done;
    k_iota<<<ceil_div(nb, T), T, 0, st>>>(idx, nb);
    int32_t* O = P + nb;
    tb = scan_temp_bytes(nb);
    if ((s = ctx->alloc(&temp, tb))) goto done;
    // phase 1: flags + scan (then the unique count is read back, untimed);
    // phase 2: zero the U outputs + segmented reduction
    cudaEvent_t e2, e3;
    GS_CUDA(cudaEventCreate(&e2));
    GS_CUDA(cudaEventCreate(&e3));
    cudaEventRecord(e0, st);
    k_run_flags<<<ceil_div(nb, T), T, 0, st>>>(keys, nb, P);
    if ((s = exclusive_scan_i32(st, P, O, nb, temp, tb))) goto done;
    cudaEventRecord(e1, st);
    int32_t* ho = (int32_t*)ctx->h_pinned;
    if (cudaMemcpyAsync(ho, O + nb - 1, 4, cudaMemcpyDeviceToHost, st) != cudaSuccess) s = GS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) s = GS_ERR_CUDA;
    *n_unique = (int64_t)ho[0] + 1;
    cudaEventRecord(e2, st);
    cudaMemsetAsync(out, 0, (size_t)*n_unique * 72, st);
    k_fast_segment_reduce<<<ceil_div(nb, T), T, 0, st>>>(keys, idx, O, blocks, nb, ~0ull, 32, out, rid, cid, koi);
    cudaEventRecord(e3, st);
    float m1 = 0.f, m2 = 0.f;
    if (cudaStreamSynchronize(st) != cudaSuccess || cudaEventElapsedTime(&m1, e0, e1) != cudaSuccess ||
        cudaEventElapsedTime(&m2, e2, e3) != cudaSuccess)
      s = GS_ERR_CUDA;
    cudaEventDestroy(e2);
    cudaEventDestroy(e3);
    *ms = m1 + m2;
  } else {
    if ((s = ctx->alloc((void**)&ukeys, (size_t)nb * 8)) || (s = ctx->alloc((void**)&nruns, 8))) goto done;
    cub::DeviceReduce::ReduceByKey(nullptr, tb, keys, ukeys, (const Block9*)blocks, (Block9*)out, nruns, Sum9(), nb,
                                   st);
    if ((s = ctx->alloc(&temp, tb))) goto done;
    cudaEventRecord(e0, st);
    cub::DeviceReduce::ReduceByKey(temp, tb, keys, ukeys, (const Block9*)blocks, (Block9*)out, nruns, Sum9(), nb,
                                   st);
    cudaEventRecord(e1, st);
    int64_t* hn = (int64_t*)ctx->h_pinned;
    if (cudaMemcpyAsync(hn, nruns, 8, cudaMemcpyDeviceToHost, st) != cudaSuccess) s = GS_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) s = GS_ERR_CUDA;
    *n_unique = hn[0];
  }
  if (s == GS_OK) {
    if (cudaGetLastError() != cudaSuccess || (method == 1 && cudaEventElapsedTime(ms, e0, e1) != cudaSuccess)) {
      set_error("gs_micro_segment_reduce: launch failed");
      s = GS_ERR_CUDA;
    }
  } else {
    set_error("gs_micro_segment_reduce: readback failed");
  }
done:
  ctx->release(temp);
  ctx->release(P);
  ctx->release(idx);
  ctx->release(rid);
  ctx->release(cid);
  ctx->release(koi);
  ctx->release(ukeys);
  ctx->release(nruns);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return s;
}
