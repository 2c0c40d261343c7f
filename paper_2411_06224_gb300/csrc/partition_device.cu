// Level-0 domain partition on the device (Sec. 3.2, Eq. num_subdomains;
// supplement Algorithm 1), the same rules as the host partition, bit for bit.
//
// GS_PART_RCB: recursive coordinate bisection of the rest positions.  The
// vertices are sorted by each coordinate once (one stable radix sort of all
// three lists); the lists are then kept grouped by set, each set in
// (coordinate, vertex index) order.  All sets of one depth are split
// together: a set's extent along an axis is the difference of the last and
// first entry of its stretch of that list, the axis of largest extent (first
// on ties) gives the side of every vertex, the first N * ceil(P / 2) going
// left, and the three lists are partitioned by side, stably, from one scan.
// New sets are numbered left before right, in set order, so the leaves come
// out numbered left to right.
//   What bounds it: launches.  The lists are 12 bytes per vertex and stay in
// L2.  Sorting all vertices by (coordinate) and by (set) at every depth and
// finding the extents by atomics took 5.9 ms at 64^3 (3.1 ms of it the
// atomics of the first depths, on a handful of addresses); now 0.5 ms.
//
// GS_PART_RCB_COMPONENTS: the same bisection started from the connected
// components of the mesh graph (numbered by their smallest vertex), found by
// hooking roots onto smaller roots with atomic minima and compressing paths
// until nothing changes; no part then mixes two bodies.
//
// GS_PART_MORTON: N consecutive vertices in Morton order (10 bits per axis
// over the bounding box, ties by vertex index), the level-0 subdomains of the
// earlier MAS the paper compares against.
//
// Finally every vertex takes slot N * part + (rank among its part's vertices
// in ascending index): a warp per part counts the smaller indices (parts of
// more than 32 vertices: a stable sort by part).
#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>

#include <algorithm>
#include <vector>

#include "common.cuh"

namespace gs {
namespace part {

// Order-preserving unsigned image of a double (-0.0 taken as +0.0, so equal
// coordinates compare equal as they do in the host rule).
__device__ __forceinline__ unsigned long long okey(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  if (b == 0x8000000000000000ull) b = 0;
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double from_okey(unsigned long long k) {
  const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
  return __longlong_as_double((long long)b);
}

__global__ void k_check_finite(const double* __restrict__ X, int64_t n3, int* __restrict__ flags) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n3 && !isfinite(X[i])) atomicOr(flags, kErrNonFinite);
}

__global__ void k_iota(int32_t* __restrict__ a, int32_t n) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = i;
}

// ---------------------------------------------------------------- components
__device__ __forceinline__ int32_t find_root(const int32_t* parent, int32_t v) {
  int32_t p = parent[v];
  while (p != v) {
    v = p;
    p = parent[v];
  }
  return v;
}

__global__ void k_hook(const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj, int32_t n,
                       int32_t* parent, int* __restrict__ changed, int* __restrict__ flags) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  for (int32_t e = adj_ptr[v]; e < adj_ptr[v + 1]; ++e) {
    const int32_t w = adj[e];
    if (w < 0 || w >= n) {
      atomicOr(flags, kErrIndex);
      continue;
    }
    const int32_t rv = find_root(parent, v), rw = find_root(parent, w);
    if (rv != rw) {
      const int32_t hi = max(rv, rw), lo = min(rv, rw);
      if (atomicMin(&parent[hi], lo) > lo) *changed = 1;
    }
  }
}

__global__ void k_compress(int32_t* parent, int32_t n) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) parent[v] = find_root(parent, v);
}

__global__ void k_root_flags(const int32_t* __restrict__ parent, int32_t n, int32_t* __restrict__ f) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) f[v] = parent[v] == v;
}

__global__ void k_label_from_roots(const int32_t* __restrict__ parent, const int32_t* __restrict__ rank, int32_t n,
                                   int32_t* __restrict__ label) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) label[v] = rank[parent[v]];
}

// ---------------------------------------------------------------- one bisection round
// Entry t of `per` lists to be sorted: vertex t % n under coordinate a0 + t / n.
__global__ void k_list_keys(const double* __restrict__ X, int32_t n, int a0, int per,
                            unsigned long long* __restrict__ key, int32_t* __restrict__ val) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)per * n) return;
  const int q = (int)(t / n);
  key[t] = okey(X[3 * (t - (int64_t)q * n) + a0 + q]);
  val[t] = (int32_t)t;
}

// Group of a sorted entry: its list, and within it its vertex's component
// (comp null: one component).
__global__ void k_list_groups(const int32_t* __restrict__ val, const int32_t* __restrict__ comp, int32_t n, int per,
                              int32_t C, uint32_t* __restrict__ group) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)per * n) return;
  const int32_t q = val[t] / n;
  group[t] = (uint32_t)(q * C + (comp ? comp[val[t] - q * n] : 0));
}

__global__ void k_list_vertices(const int32_t* __restrict__ val, int32_t n, int per, int32_t* __restrict__ list) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (int64_t)per * n) list[t] = val[t] % n;
}

// Set of every position (its vertex's component), and the first position and
// size of every set.
__global__ void k_list_init(const int32_t* __restrict__ list, const int32_t* __restrict__ comp, int32_t n,
                            int32_t* __restrict__ pset, int32_t* __restrict__ start, int32_t* __restrict__ size,
                            int32_t* __restrict__ largest) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int32_t s = comp ? comp[list[p]] : 0;
  pset[p] = s;
  if (p > 0 && (!comp || comp[list[p - 1]] == s)) return;
  start[s] = p;
  int32_t lo = p + 1, hi = n;  // the stretch ends at the first position of a larger component
  while (comp && lo < hi) {
    const int32_t mid = lo + (hi - lo) / 2;
    if (comp[list[mid]] == s)
      lo = mid + 1;
    else
      hi = mid;
  }
  size[s] = hi - p;
  atomicMax(largest, hi - p);
}

// Per set: axis of largest extent (first on ties, the extents computed in
// double as max - min), whether it splits, its left size.  *count sets exist,
// the launch covers `bound` of them.
__global__ void k_set_plan(const int32_t* __restrict__ count, int32_t bound, int N, const double* __restrict__ X,
                           const int32_t* __restrict__ list, int32_t n, const int32_t* __restrict__ start,
                           const int32_t* __restrict__ size, int8_t* __restrict__ axis, int32_t* __restrict__ width,
                           int32_t* __restrict__ left) {
  const int32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s > bound) return;
  if (s >= *count) {
    width[s] = 0;
    return;
  }
  const int32_t p0 = start[s], p1 = p0 + size[s] - 1;
  int best = 0;
  double ext = 0.0;
  for (int a = 0; a < 3; ++a) {
    const int64_t o = (int64_t)a * n;
    const double e = X[3 * (int64_t)list[o + p1] + a] - X[3 * (int64_t)list[o + p0] + a];
    if (a == 0 || e > ext) ext = e, best = a;
  }
  axis[s] = (int8_t)best;
  const int32_t P = (size[s] + N - 1) / N;
  width[s] = P > 1 ? 2 : 1;
  left[s] = N * ((P + 1) / 2);
}

// Side of every vertex (by its position in the list of its set's axis), and
// the new sets: ids first[s], first[s] + 1.
__global__ void k_set_sides(const int32_t* __restrict__ list, int32_t n, const int32_t* __restrict__ pset,
                            const int32_t* __restrict__ start, const int32_t* __restrict__ size,
                            const int8_t* __restrict__ axis, const int32_t* __restrict__ width,
                            const int32_t* __restrict__ left, const int32_t* __restrict__ first, int32_t bound,
                            const int32_t* __restrict__ count, uint8_t* __restrict__ side, int32_t* __restrict__ start2,
                            int32_t* __restrict__ size2, int32_t* __restrict__ count2) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  if (p == 0) *count2 = first[bound];
  const int32_t s = pset[p];
  side[list[(int64_t)axis[s] * n + p]] = width[s] == 2 && p - start[s] >= left[s];
  if (p < *count) {
    const int32_t f = first[p], two = width[p] == 2;
    start2[f] = start[p];
    size2[f] = two ? left[p] : size[p];
    if (two) start2[f + 1] = start[p] + left[p], size2[f + 1] = size[p] - left[p];
  }
}

__global__ void k_left_flags(const int32_t* __restrict__ list, int32_t n, const uint8_t* __restrict__ side,
                             uint32_t* __restrict__ f) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < 3LL * n) f[t] = side[list[t]] == 0;
}

// Stable partition of the three lists by side inside every set; before[]: the
// exclusive scan of the left flags (modulo 2^32: only differences count).
__global__ void k_list_split(const int32_t* __restrict__ list, int32_t n, const uint32_t* __restrict__ before,
                             const uint8_t* __restrict__ side, const int32_t* __restrict__ pset,
                             const int32_t* __restrict__ start, const int32_t* __restrict__ width,
                             const int32_t* __restrict__ left, const int32_t* __restrict__ first,
                             int32_t* __restrict__ list2, int32_t* __restrict__ pset2) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 3LL * n) return;
  const int64_t o = t / n * n;
  const int32_t p = (int32_t)(t - o), s = pset[p], p0 = start[s], v = list[t];
  const int32_t nl = (int32_t)(before[t] - before[o + p0]);
  list2[o + (side[v] ? p0 + left[s] + (p - p0 - nl) : p0 + nl)] = v;
  if (o == 0) pset2[p] = first[s] + (width[s] == 2 && p - p0 >= left[s] ? 1 : 0);
}

// ---------------------------------------------------------------- Morton order
__global__ void k_box(const double* __restrict__ X, int32_t n, unsigned long long* __restrict__ lo,
                      unsigned long long* __restrict__ hi) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  for (int a = 0; a < 3; ++a) {
    const unsigned long long k = okey(X[3 * (int64_t)v + a]);
    atomicMin(&lo[a], k);
    atomicMax(&hi[a], k);
  }
}

constexpr int kMortonBits = 10;

__global__ void k_morton(const double* __restrict__ X, int32_t n, const unsigned long long* __restrict__ lo,
                         const unsigned long long* __restrict__ hi, uint32_t* __restrict__ code) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= n) return;
  uint32_t c = 0;
  for (int a = 0; a < 3; ++a) {
    const double l = from_okey(lo[a]), e = from_okey(hi[a]) - l;
    uint32_t q = 0;
    if (e > 0.0) {
      // the host rule's arithmetic, operation for operation (no contraction)
      const double t = __dmul_rn(__ddiv_rn(__dsub_rn(X[3 * (int64_t)v + a], l), e), (double)(1 << kMortonBits));
      q = (uint32_t)min(floor(t), (double)((1 << kMortonBits) - 1));
    }
    for (int b = 0; b < kMortonBits; ++b) c |= ((q >> b) & 1u) << (3 * b + a);
  }
  code[v] = c;
}

__global__ void k_morton_sets(int32_t n, int N, int32_t* __restrict__ pset, int32_t* __restrict__ start,
                              int32_t* __restrict__ size) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  pset[p] = p / N;
  if (p % N == 0) start[p / N] = p, size[p / N] = min(N, n - p);
}

// ---------------------------------------------------------------- slots
// Parts of at most 32 vertices: a warp per part; a vertex's rank is the number
// of the part's vertices with a smaller index.
__global__ void k_slots_warp(const int32_t* __restrict__ list, const int32_t* __restrict__ start,
                             const int32_t* __restrict__ size, int32_t parts, int N, int32_t* __restrict__ map,
                             int* __restrict__ flags) {
  const int32_t q = (int32_t)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (q >= parts) return;  // whole warp
  const int32_t m = size[q];
  if (m > N) {  // a part larger than the domain size (not reachable)
    if (lane == 0) atomicOr(flags, kErrIndex);
    return;
  }
  const int32_t v = lane < m ? list[start[q] + lane] : INT32_MAX;
  int32_t rank = 0;
#pragma unroll
  for (int k = 0; k < 32; ++k) rank += __shfl_sync(0xffffffffu, v, k) < v;
  if (lane < m) map[v] = q * N + rank;
}

// Longer parts: from the vertices sorted by (part, index).
__global__ void k_part_labels(const int32_t* __restrict__ list, const int32_t* __restrict__ pset, int32_t n,
                              int32_t* __restrict__ label) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) label[list[p]] = pset[p];
}

__global__ void k_slots(const int32_t* __restrict__ order, int32_t n, const int32_t* __restrict__ label,
                        const int32_t* __restrict__ start, int N, int32_t* __restrict__ map, int* __restrict__ flags) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int32_t v = order[p];
  const int32_t q = label[v];
  const int32_t rank = p - start[q];
  if (rank >= N) atomicOr(flags, kErrIndex);  // a part larger than the domain size (not reachable)
  map[v] = q * N + rank;
}

}  // namespace part

namespace {

// Device buffers of one partition call, freed on every return.
struct Tmp {
  gs_ctx ctx;
  std::vector<void*> ptrs;
  ~Tmp() {
    for (void* p : ptrs) ctx->release(p);
  }
  template <typename T>
  int get(T** out, size_t count) {
    void* p = nullptr;
    GS_TRY(ctx->alloc(&p, std::max<size_t>(count, 1) * sizeof(T)));
    ptrs.push_back(p);
    *out = (T*)p;
    return GS_OK;
  }
};

int read_int(gs_ctx ctx, const int32_t* d, int32_t* h) {
  GS_CUDA(cudaMemcpyAsync(ctx->h_pinned + 8, d, 4, cudaMemcpyDeviceToHost, ctx->stream));
  GS_CUDA(cudaStreamSynchronize(ctx->stream));
  *h = ctx->h_pinned[8];
  return GS_OK;
}

int exclusive_sum(gs_ctx ctx, Tmp& tmp, const int32_t* in, int32_t* out, int32_t count) {
  size_t tb = 0;
  GS_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, in, out, count, ctx->stream));
  void* t;
  GS_TRY(tmp.get((char**)&t, tb));
  GS_PROF(ctx, GS_K_LIBPRIM);
  GS_CUDA(cub::DeviceScan::ExclusiveSum(t, tb, in, out, count, ctx->stream));
  return GS_OK;
}

template <typename K>
int sort_pairs(gs_ctx ctx, Tmp& tmp, const K* kin, K* kout, const int32_t* vin, int32_t* vout, int32_t count,
               int end_bit) {
  size_t tb = 0;
  GS_CUDA(cub::DeviceRadixSort::SortPairs(nullptr, tb, kin, kout, vin, vout, count, 0, end_bit, ctx->stream));
  void* t;
  GS_TRY(tmp.get((char**)&t, tb));
  GS_PROF(ctx, GS_K_LIBPRIM);
  GS_CUDA(cub::DeviceRadixSort::SortPairs(t, tb, kin, kout, vin, vout, count, 0, end_bit, ctx->stream));
  return GS_OK;
}

}  // namespace

// The parts of the vertices by `rule` (GS_PART_*): *list holds the vertices
// grouped by part, part q at (*start)[q] with (*size)[q] of them; *n_parts on
// the host; (*pset)[p] is the part of list entry p.  The arrays live in tmp.
static int partition_parts(gs_ctx ctx, Tmp& tmp, int32_t n, const double* X, const int32_t* adj_ptr, const int32_t* adj,
                           int32_t N, int32_t rule, int32_t** out_list, int32_t** out_pset, int32_t** out_start,
                           int32_t** out_size, int32_t* n_parts) {
  using namespace part;
  cudaStream_t st = ctx->stream;
  const int gv = ceil_div(n, 256), g3 = ceil_div(3LL * n, 256);
  int flags = 0;
  { GS_PROF(ctx, GS_K_OTHER); k_check_finite<<<g3, 256, 0, st>>>(X, 3LL * n, ctx->d_flags); }
  GS_TRY(ctx->take_flags(&flags));
  GS_CHECK(!flags, GS_ERR_INVALID, "partition: non-finite position");

  if (rule == GS_PART_MORTON) {
    int32_t *order, *iota, *pset, *start, *size;
    unsigned long long* box;
    uint32_t *code, *code2;
    const int32_t parts = (int32_t)(((int64_t)n + N - 1) / N);
    GS_TRY(tmp.get(&order, n));
    GS_TRY(tmp.get(&iota, n));
    GS_TRY(tmp.get(&pset, n));
    GS_TRY(tmp.get(&start, parts));
    GS_TRY(tmp.get(&size, parts));
    GS_TRY(tmp.get(&box, 6));
    GS_TRY(tmp.get(&code, n));
    GS_TRY(tmp.get(&code2, n));
    { GS_PROF(ctx, GS_K_OTHER); k_iota<<<gv, 256, 0, st>>>(iota, n); }
    GS_CUDA(cudaMemsetAsync(box, 0xff, 3 * 8, st));
    GS_CUDA(cudaMemsetAsync(box + 3, 0, 3 * 8, st));
    { GS_PROF(ctx, GS_K_OTHER); k_box<<<gv, 256, 0, st>>>(X, n, box, box + 3); }
    { GS_PROF(ctx, GS_K_OTHER); k_morton<<<gv, 256, 0, st>>>(X, n, box, box + 3, code); }
    GS_TRY(sort_pairs(ctx, tmp, code, code2, iota, order, n, 3 * kMortonBits));
    { GS_PROF(ctx, GS_K_OTHER); k_morton_sets<<<gv, 256, 0, st>>>(n, N, pset, start, size); }
    GS_CUDA(cudaGetLastError());
    *out_list = order, *out_pset = pset, *out_start = start, *out_size = size, *n_parts = parts;
    return GS_OK;
  }

  int32_t S = 1;
  int32_t* comp = nullptr;  // component of every vertex
  if (rule == GS_PART_RCB_COMPONENTS) {
    GS_CHECK(adj_ptr && adj, GS_ERR_INVALID, "partition: the component rule needs the mesh graph");
    int32_t *parent, *rootf, *rank;
    GS_TRY(tmp.get(&parent, n));
    GS_TRY(tmp.get(&rootf, n + 1));
    GS_TRY(tmp.get(&rank, n + 1));
    GS_TRY(tmp.get(&comp, n));
    int* changed = ctx->d_flags + 32;
    { GS_PROF(ctx, GS_K_OTHER); k_iota<<<gv, 256, 0, st>>>(parent, n); }
    for (int round = 0;; ++round) {
      GS_CHECK(round < 64 * 1024, GS_ERR_INVALID, "partition: components did not settle");
      GS_CUDA(cudaMemsetAsync(changed, 0, 4, st));
      { GS_PROF(ctx, GS_K_OTHER); k_hook<<<gv, 256, 0, st>>>(adj_ptr, adj, n, parent, changed, ctx->d_flags); }
      { GS_PROF(ctx, GS_K_OTHER); k_compress<<<gv, 256, 0, st>>>(parent, n); }
      int32_t ch = 0;
      GS_TRY(read_int(ctx, changed, &ch));
      if (!ch) break;
    }
    GS_TRY(ctx->take_flags(&flags));
    GS_CHECK(!flags, GS_ERR_INVALID, "partition: a neighbour index is out of range");
    GS_CUDA(cudaMemsetAsync(rootf + n, 0, 4, st));
    { GS_PROF(ctx, GS_K_OTHER); k_root_flags<<<gv, 256, 0, st>>>(parent, n, rootf); }
    GS_TRY(exclusive_sum(ctx, tmp, rootf, rank, n + 1));
    GS_TRY(read_int(ctx, rank + n, &S));
    { GS_PROF(ctx, GS_K_OTHER); k_label_from_roots<<<gv, 256, 0, st>>>(parent, rank, n, comp); }
  }

  // The three lists, sorted by (component, coordinate, index): one stable sort
  // of all their entries by coordinate and one by list and component (a list
  // at a time where the entries would not fit 31 bits).
  const int64_t n3 = 3LL * n;
  const int per = n3 < (1LL << 31) ? 3 : 1;
  const int64_t np = (int64_t)per * n;
  int32_t *list, *list2;
  GS_TRY(tmp.get(&list, n3));
  GS_TRY(tmp.get(&list2, n3));
  {
    Tmp sort_tmp{ctx};
    unsigned long long *key, *key2;
    int32_t *val, *val2;
    GS_TRY(sort_tmp.get(&key, np));
    GS_TRY(sort_tmp.get(&key2, np));
    GS_TRY(sort_tmp.get(&val, np));
    GS_TRY(sort_tmp.get(&val2, np));
    const int gp = ceil_div(np, 256);
    for (int a0 = 0; a0 < 3; a0 += per) {
      { GS_PROF(ctx, GS_K_OTHER); k_list_keys<<<gp, 256, 0, st>>>(X, n, a0, per, key, val); }
      GS_TRY(sort_pairs(ctx, sort_tmp, key, key2, val, val2, (int32_t)np, 64));
      if ((int64_t)per * S > 1) {
        uint32_t *grp = (uint32_t*)key, *grp2 = (uint32_t*)key2;
        { GS_PROF(ctx, GS_K_OTHER); k_list_groups<<<gp, 256, 0, st>>>(val2, comp, n, per, S, grp); }
        GS_TRY(sort_pairs(ctx, sort_tmp, grp, grp2, val2, val, (int32_t)np, bits_for((int64_t)per * S - 1)));
        std::swap(val, val2);
      }
      { GS_PROF(ctx, GS_K_OTHER); k_list_vertices<<<gp, 256, 0, st>>>(val2, n, per, list + (int64_t)a0 * n); }
    }
  }
  // at most this many sets ever exist: each set ends in at least one part
  const int32_t cap = (int32_t)std::min<int64_t>(n, (int64_t)S + n / N);
  int32_t *pset, *pset2, *start, *start2, *size, *size2, *width, *first, *left, *word;
  uint32_t* before;
  int8_t* axis;
  uint8_t* side;
  GS_TRY(tmp.get(&pset, n));
  GS_TRY(tmp.get(&pset2, n));
  GS_TRY(tmp.get(&start, cap));
  GS_TRY(tmp.get(&start2, cap));
  GS_TRY(tmp.get(&size, cap));
  GS_TRY(tmp.get(&size2, cap));
  GS_TRY(tmp.get(&width, cap + 1));
  GS_TRY(tmp.get(&first, cap + 1));
  GS_TRY(tmp.get(&left, cap));
  GS_TRY(tmp.get(&axis, cap));
  GS_TRY(tmp.get(&side, n));
  GS_TRY(tmp.get(&before, n3));
  GS_TRY(tmp.get(&word, 4));  // set counts of this depth and the next; the largest component
  int32_t *count = word, *count2 = word + 1, *largest = word + 2;
  GS_CUDA(cudaMemsetAsync(largest, 0, 4, st));
  GS_CUDA(cudaMemcpyAsync(count, &S, 4, cudaMemcpyHostToDevice, st));
  { GS_PROF(ctx, GS_K_OTHER); k_list_init<<<gv, 256, 0, st>>>(list, comp, n, pset, start, size, largest); }
  int32_t most = n;
  if (comp) GS_TRY(read_int(ctx, largest, &most));
  size_t tb = 0, tb3 = 0;
  GS_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb, width, first, cap + 1, st));
  GS_CUDA(cub::DeviceScan::ExclusiveSum(nullptr, tb3, before, before, n3, st));
  char* temp;
  tb = std::max(tb, tb3);
  GS_TRY(tmp.get(&temp, tb));
  // ceil(P / 2) parts go left, so a set of P parts is split up after
  // ceil(log2 P) depths; the host needs no count in between
  int32_t bound = S;
  for (int64_t P = ((int64_t)most + N - 1) / N; P > 1; P = (P + 1) / 2) {
    { GS_PROF(ctx, GS_K_OTHER); k_set_plan<<<ceil_div(bound + 1, 256), 256, 0, st>>>(count, bound, N, X, list, n, start, size, axis, width, left); }
    { GS_PROF(ctx, GS_K_LIBPRIM); GS_CUDA(cub::DeviceScan::ExclusiveSum(temp, tb, width, first, bound + 1, st)); }
    { GS_PROF(ctx, GS_K_OTHER); k_set_sides<<<gv, 256, 0, st>>>(list, n, pset, start, size, axis, width, left, first, bound, count, side, start2,
                                                                size2, count2); }
    { GS_PROF(ctx, GS_K_OTHER); k_left_flags<<<g3, 256, 0, st>>>(list, n, side, before); }
    { GS_PROF(ctx, GS_K_LIBPRIM); GS_CUDA(cub::DeviceScan::ExclusiveSum(temp, tb, before, before, n3, st)); }
    { GS_PROF(ctx, GS_K_OTHER); k_list_split<<<g3, 256, 0, st>>>(list, n, before, side, pset, start, width, left, first, list2, pset2); }
    std::swap(list, list2);
    std::swap(pset, pset2);
    std::swap(start, start2);
    std::swap(size, size2);
    std::swap(count, count2);
    bound = (int32_t)std::min<int64_t>(2LL * bound, cap);
  }
  GS_CUDA(cudaGetLastError());
  GS_TRY(read_int(ctx, count, n_parts));
  *out_list = list, *out_pset = pset, *out_start = start, *out_size = size;
  return GS_OK;
}

}  // namespace gs

extern "C" int gs_partition_device(gs_ctx ctx, int32_t n, const double* X, const int32_t* adj_ptr,
                                   const int32_t* adj, int32_t N, int32_t rule, int32_t* map, int32_t* n_domains) {
  using namespace gs;
  GS_CHECK(ctx && X && map && n_domains, GS_ERR_INVALID, "gs_partition_device: null argument");
  GS_CHECK(n >= 1 && N >= 1, GS_ERR_INVALID, "gs_partition_device: n %d, domain size %d", n, N);
  GS_CHECK(rule == GS_PART_RCB || rule == GS_PART_RCB_COMPONENTS || rule == GS_PART_MORTON, GS_ERR_INVALID,
           "gs_partition_device: rule %d", rule);
  GS_CUDA(cudaSetDevice(ctx->device));
  Tmp tmp{ctx};
  cudaStream_t st = ctx->stream;
  int32_t *list, *pset, *start, *size, M = 0;
  GS_TRY(partition_parts(ctx, tmp, n, X, adj_ptr, adj, N, rule, &list, &pset, &start, &size, &M));
  if (N <= 32) {
    GS_PROF(ctx, GS_K_OTHER);
    part::k_slots_warp<<<ceil_div(32LL * M, 256), 256, 0, st>>>(list, start, size, M, N, map, ctx->d_flags);
  } else {
    int32_t *label, *lab_sorted, *iota, *order;
    GS_TRY(tmp.get(&label, n));
    GS_TRY(tmp.get(&lab_sorted, n));
    GS_TRY(tmp.get(&iota, n));
    GS_TRY(tmp.get(&order, n));
    const int gv = ceil_div(n, 256);
    { GS_PROF(ctx, GS_K_OTHER); part::k_iota<<<gv, 256, 0, st>>>(iota, n); }
    { GS_PROF(ctx, GS_K_OTHER); part::k_part_labels<<<gv, 256, 0, st>>>(list, pset, n, label); }
    GS_TRY(sort_pairs(ctx, tmp, label, lab_sorted, iota, order, n, bits_for(M)));  // by part, ties by index
    { GS_PROF(ctx, GS_K_OTHER); part::k_slots<<<gv, 256, 0, st>>>(order, n, label, start, N, map, ctx->d_flags); }
  }
  int flags = 0;
  GS_TRY(ctx->take_flags(&flags));
  if (flags) return status_from_flags(flags);
  *n_domains = M;
  return GS_OK;
}

extern "C" int gs_build_mas_mesh(gs_ctx ctx, gs_mat mat, const double* X, int32_t part_rule, const int32_t* adj_ptr,
                                 const int32_t* adj, const int32_t* contacts, int64_t n_contacts,
                                 const gs_mas_opts* opts, gs_mas* out) {
  using namespace gs;
  GS_CHECK(ctx && mat && X && opts && out, GS_ERR_INVALID, "gs_build_mas_mesh: null argument");
  GS_CUDA(cudaSetDevice(ctx->device));
  int32_t* map = nullptr;
  GS_TRY(ctx->alloc((void**)&map, (size_t)std::max(mat->n, 1) * 4));
  int32_t nd = 0;
  int s = gs_partition_device(ctx, mat->n, X, adj_ptr, adj, opts->domain_size, part_rule, map, &nd);
  if (s == GS_OK) s = gs_build_mas(ctx, mat, map, nd, adj_ptr, adj, contacts, n_contacts, opts, out);
  ctx->release(map);
  return s;
}
