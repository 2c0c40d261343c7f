// Batched PCG over independent systems (this library's batching form; the
// paper solves one system at a time).
//
// The systems are the diagonal blocks of one block-diagonal matrix: system s
// owns block rows [node_off[s], node_off[s+1]).  Assembled and preconditioned
// as one matrix -- each system partitioned on its own, so no level-0 domain
// and, having no edges between systems, no supernode mixes two systems --
// they share every SpMV and MAS-apply launch, while PCG keeps one recurrence
// per system: vectors are cut into (system, chunk) work items, four blocks each, a
// reduction writes one partial sum per block, and every block that needs a
// system's scalar adds that system's partials in the same fixed order, so the
// result is deterministic; alpha, beta and the convergence test are per system.
// A converged system stops moving.
// 24 bodies, 188,000 block rows: an iteration took 302 us, 24 of them a dot
// product and 26 the x, r update (one load in flight per thread, the last block's
// sums); 239 now, 164 of them the two products.
//
// The iteration loop can run inside one CUDA graph: a conditional WHILE node
// whose body is one PCG iteration and whose last kernel clears the condition
// once every system converged or max_iter iterations ran, so a whole batched
// solve is one graph launch with no host round trip.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "pcg_state.cuh"
#include "primitives.cuh"

namespace gs {

int spmv_launch(gs_ctx ctx, gs_mat m, const double* x, double* y, int nrhs, int variant);
int mas_apply_launch(gs_ctx ctx, gs_mas mas, const double* r, double* z, int nrhs, double* rl, double* zl);
int mas_level_vectors(gs_ctx ctx, gs_mas mas, int nrhs, double** rl, double** zl);
bool mas_dot_usable(gs_ctx ctx, gs_mas mas, int nrhs);
int mas_restrict(gs_ctx ctx, gs_mas mas, const double* r, int nrhs, double* rl, const int* skip);
int mas_products(gs_ctx ctx, gs_mas mas, const double* r, double* z, int nrhs, double* rl, double* zl, const int* skip,
                 const Partials* dot);
int ensure_row_order(gs_ctx ctx, gs_mat m);

namespace batch {

constexpr int kT = 256;
constexpr int kLoads = 4;  // entries per thread whose loads are in flight together
constexpr int kParts = 4;  // blocks per work item: 141 items of 4096 entries are less than a block per SM

struct Head {  // per-batch control words (device)
  int all_conv;
  int running;  // systems that have not converged
  int flags;
  int iter;  // iterations run (graph mode)
};

struct Arrays {  // per-system scalars (device arrays of length S)
  double *bnorm2, *rz, *rz_old, *rr;  // rz: r . z of the iteration to come; rz_old: the one its alpha was taken with
  int *conv, *bad, *iters;
  double *pap, *rrp, *rzp;  // partial sums, kParts per work item
  const int32_t *w_seg;     // work item -> system
  const int64_t *w_beg, *w_end;
  const int32_t* w_start;  // system -> first work item (S + 1 entries)
  int S;
};

__device__ __forceinline__ double block_sum(double v) {  // valid in thread 0
  __shared__ double red[kT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = warp_sum(v);
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0)
#pragma unroll
    for (int i = 1; i < kT / 32; ++i) v += red[i];
  return v;
}

// This block's quarter of its work item.
struct Span {
  int w, at;  // item, place of its partial sum
  int64_t beg, end;
};
__device__ __forceinline__ Span my_span(const Arrays& a) {
  const int w = blockIdx.x, part = blockIdx.y;
  const int64_t b = a.w_beg[w], e = a.w_end[w], per = (e - b + kParts - 1) / kParts;
  return Span{w, w * kParts + part, min(b + part * per, e), min(b + (part + 1) * per, e)};
}

// Sum of a system's partials by a warp.
__device__ __forceinline__ double system_sum(const double* part, const Arrays& a, int s) {
  Partials q;
  q.sum = const_cast<double*>(part) + kParts * a.w_start[s];
  q.n = kParts * (a.w_start[s + 1] - a.w_start[s]);
  return warp_sum_partials(q, 0);
}

// r = b, x = 0, partial sums of ||b||^2.
__global__ void __launch_bounds__(kT) k_binit(const double* __restrict__ b, double* __restrict__ x,
                                              double* __restrict__ r, Arrays a) {
  const Span sp = my_span(a);
  const int64_t end = sp.end;
  double v = 0.0;
  for (int64_t i = sp.beg + threadIdx.x; i < end; i += kT * kLoads) {
    double q[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) q[u] = i + u * kT < end ? b[i + u * kT] : 0.0;
#pragma unroll
    for (int u = 0; u < kLoads; ++u)
      if (i + u * kT < end) {
        x[i + u * kT] = 0.0;
        r[i + u * kT] = q[u];
        v = fma(q[u], q[u], v);
      }
  }
  v = block_sum(v);
  if (threadIdx.x == 0) a.rrp[sp.at] = v;
}

// Partial sums of u . v; kCopy also writes dst = v.
template <bool kCopy>
__global__ void __launch_bounds__(kT) k_bdot(const double* u_, const double* v_, double* __restrict__ dst,
                                             const Head* h, Arrays a, double* __restrict__ out) {
  wait_for_previous_kernel();
  if (!kCopy && h->all_conv) return;
  const Span sp = my_span(a);
  const int64_t end = sp.end;
  double v = 0.0;
  for (int64_t i = sp.beg + threadIdx.x; i < end; i += kT * kLoads) {
    double p[kLoads], q[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const bool in = i + u * kT < end;
      p[u] = in ? u_[i + u * kT] : 0.0;
      q[u] = in ? v_[i + u * kT] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u)
      if (i + u * kT < end) {
        v = fma(p[u], q[u], v);
        if (kCopy) dst[i + u * kT] = q[u];
      }
  }
  let_next_kernel_launch();
  v = block_sum(v);
  if (threadIdx.x == 0) out[sp.at] = v;
}

// The first scalars, a warp per system (Head is zeroed).
__global__ void __launch_bounds__(32) k_bfirst(Head* h, Arrays a) {
  const int s = blockIdx.x;
  const double b2 = system_sum(a.rrp, a, s), rz = system_sum(a.rzp, a, s);
  if (threadIdx.x != 0) return;
  const bool finite = isfinite(b2) && isfinite(rz);
  if (!finite) atomicOr(&h->flags, kErrNonFinite);
  a.bnorm2[s] = a.rr[s] = b2;
  a.rz[s] = rz;
  a.bad[s] = a.iters[s] = 0;
  a.conv[s] = !finite || b2 == 0.0;
  if (!a.conv[s]) atomicAdd(&h->running, 1);
}
__global__ void k_bfirst_running(Head* h) { h->all_conv = h->running == 0; }

// alpha from the partial sums of p . Ap; x += alpha p, r -= alpha Ap and partial
// sums of ||r||^2.  The system's first block keeps what the sums decide; the
// others may read conv and bad before or after, the answer is the same.
__global__ void __launch_bounds__(kT) k_bupdate_xr(double* __restrict__ x, double* __restrict__ r,
                                                   const double* p, const double* Ap, Head* h, Arrays a) {
  wait_for_previous_kernel();
  if (h->all_conv) return;
  __shared__ double s_alpha;
  const Span sp = my_span(a);
  const int s = a.w_seg[sp.w];
  if (threadIdx.x < 32) {
    const double sum = system_sum(a.pap, a, s);
    if (threadIdx.x == 0) {
      const bool record = sp.at == kParts * a.w_start[s], stopped = a.conv[s] || a.bad[s];
      const bool ok = sum > 0.0 && isfinite(sum);
      if (record && !stopped && !ok) {
        atomicOr(&h->flags, isfinite(sum) ? kErrNotSPD : kErrNonFinite);
        a.bad[s] = 1;
      }
      const double rz = a.rz[s];
      if (record) a.rz_old[s] = rz;
      s_alpha = stopped || !ok ? 0.0 : rz / sum;
    }
  }
  __syncthreads();
  const double al = s_alpha;
  const int64_t end = sp.end;
  double v = 0.0;
  for (int64_t i = sp.beg + threadIdx.x; i < end; i += kT * kLoads) {
    double rv[kLoads], xv[kLoads], pv[kLoads], av[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int64_t j = i + u * kT;
      rv[u] = j < end ? r[j] : 0.0;
      xv[u] = pv[u] = av[u] = 0.0;
      if (al != 0.0 && j < end) xv[u] = x[j], pv[u] = p[j], av[u] = Ap[j];
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const int64_t j = i + u * kT;
      if (j >= end) continue;
      if (al != 0.0) {
        x[j] = fma(al, pv[u], xv[u]);
        rv[u] = fma(-al, av[u], rv[u]);
        r[j] = rv[u];
      }
      v = fma(rv[u], rv[u], v);
    }
  }
  let_next_kernel_launch();
  v = block_sum(v);
  if (threadIdx.x == 0) a.rrp[sp.at] = v;
}

// The convergence test from the partial sums of ||r||^2, beta from those of
// r . z, and p = z + beta p.
__global__ void __launch_bounds__(kT) k_bupdate_p(double* __restrict__ p, const double* z, Head* h, Arrays a,
                                                  double tol2) {
  wait_for_previous_kernel();
  __shared__ double s_beta;
  __shared__ int s_stop;
  const Span sp = my_span(a);
  const int s = a.w_seg[sp.w];
  if (threadIdx.x < 32) {
    // all_conv is read once for the block: this grid's recording blocks may set it
    const bool over = __shfl_sync(kFull, threadIdx.x == 0 ? h->all_conv : 0, 0) != 0;
    const double rr = over ? 0.0 : system_sum(a.rrp, a, s), rz = over ? 0.0 : system_sum(a.rzp, a, s);
    if (over) {
      if (threadIdx.x == 0) s_stop = 1;
    } else if (threadIdx.x == 0) {
      const bool record = sp.at == kParts * a.w_start[s];
      const bool was = a.conv[s] != 0, bad = a.bad[s] != 0 || !isfinite(rr);
      const bool stop = was || bad || rr <= tol2 * a.bnorm2[s];
      s_beta = rz / a.rz_old[s];
      s_stop = stop;
      if (record && !was) {
        if (!isfinite(rr)) {
          atomicOr(&h->flags, kErrNonFinite);
        } else if (!bad) {
          a.rr[s] = rr;
          a.iters[s] += 1;
        }
        if (!stop && !isfinite(rz)) {
          atomicOr(&h->flags, kErrNonFinite);
          a.bad[s] = 1;
        }
        a.rz[s] = rz;
        if (stop) {
          a.conv[s] = 1;
          if (atomicSub(&h->running, 1) == 1) h->all_conv = 1;
        }
      }
    }
  }
  __syncthreads();
  if (s_stop) return;
  const double be = s_beta;
  const int64_t end = sp.end;
  for (int64_t i = sp.beg + threadIdx.x; i < end; i += kT * kLoads) {
    double pv[kLoads], zv[kLoads];
#pragma unroll
    for (int u = 0; u < kLoads; ++u) {
      const bool in = i + u * kT < end;
      pv[u] = in ? p[i + u * kT] : 0.0;
      zv[u] = in ? z[i + u * kT] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kLoads; ++u)
      if (i + u * kT < end) p[i + u * kT] = fma(be, pv[u], zv[u]);
  }
  let_next_kernel_launch();
}

// Last kernel of a graph iteration: keep looping while some system runs and
// fewer than max_iter iterations have been done (the loop always ends).
__global__ void k_loop_condition(cudaGraphConditionalHandle cond, Head* h, int max_iter) {
  const int it = ++h->iter;
  cudaGraphSetConditional(cond, (!h->all_conv && !h->flags && it < max_iter) ? 1u : 0u);
}

}  // namespace batch

extern "C" int gs_pcg_solve_batch(gs_ctx ctx, gs_mat mat, gs_mas mas, int32_t n_sys, const int32_t* node_off,
                                  const double* b, double tol, int32_t max_iter, int32_t use_graph, double* x,
                                  int32_t* iters, double* rel_res) {
  using namespace batch;
  GS_CHECK(ctx && mat && mas && node_off && b && x && b != x, GS_ERR_INVALID, "gs_pcg_solve_batch: null argument");
  GS_CHECK(n_sys >= 1, GS_ERR_INVALID, "gs_pcg_solve_batch: n_sys %d", n_sys);
  GS_CHECK(mas->n == mat->n && node_off[0] == 0 && node_off[n_sys] == mat->n, GS_ERR_INVALID,
           "gs_pcg_solve_batch: node offsets do not span the matrix");
  for (int s = 0; s < n_sys; ++s)
    GS_CHECK(node_off[s + 1] >= node_off[s], GS_ERR_INVALID, "gs_pcg_solve_batch: offsets not ascending");
  GS_CHECK(tol >= 0.0 && max_iter >= 0, GS_ERR_INVALID, "gs_pcg_solve_batch: tol %g max_iter %d", tol, max_iter);
  GS_CUDA(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  const int64_t len = 3LL * mat->n;
  // work list: chunks of every system's entries, in system order
  const int64_t kChunk = ctx->tune[GS_TUNE_BATCH_CHUNK];
  std::vector<int32_t> w_seg, w_start(n_sys + 1);
  std::vector<int64_t> w_beg, w_end;
  for (int s = 0; s < n_sys; ++s) {
    w_start[s] = (int32_t)w_seg.size();
    const int64_t b0 = 3LL * node_off[s], b1 = 3LL * node_off[s + 1];
    for (int64_t c = b0; c < b1; c += kChunk) {
      w_seg.push_back(s);
      w_beg.push_back(c);
      w_end.push_back(std::min(c + kChunk, b1));
    }
  }
  w_start[n_sys] = (int32_t)w_seg.size();
  if (w_seg.empty()) {  // all systems empty
    w_seg.push_back(0), w_beg.push_back(0), w_end.push_back(0);
  }
  const int W = (int)w_seg.size();
  // device buffers: vectors r, z, p, Ap; scalars; work list; partials
  double* vec = nullptr;
  GS_TRY(ctx->scratch_buf(kSlotPcgVectors, 4 * (size_t)len * sizeof(double) + 64, (void**)&vec));
  double *r = vec, *z = r + len, *p = z + len, *Ap = p + len;
  auto r256 = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t sz = r256(sizeof(Head)) + 4 * r256((size_t)n_sys * 8) + 3 * r256((size_t)n_sys * 4) +
                    r256((size_t)W * 4) + 2 * r256((size_t)W * 8) + r256((size_t)(n_sys + 1) * 4) +
                    3 * r256((size_t)W * kParts * 8) + 256;
  char* buf = nullptr;
  GS_TRY(ctx->scratch_buf(kSlotPcgScalars, sz, (void**)&buf));
  auto take = [&](size_t bytes) {
    char* q = buf;
    buf += (bytes + 255) / 256 * 256;
    return q;
  };
  Head* h = (Head*)take(sizeof(Head));
  Arrays a{};
  a.S = n_sys;
  a.bnorm2 = (double*)take(n_sys * 8);
  a.rz = (double*)take(n_sys * 8);
  a.rz_old = (double*)take(n_sys * 8);
  a.rr = (double*)take(n_sys * 8);
  a.conv = (int*)take(n_sys * 4);
  a.bad = (int*)take(n_sys * 4);
  a.iters = (int*)take(n_sys * 4);
  int32_t* d_wseg = (int32_t*)take(W * 4);
  int64_t* d_wbeg = (int64_t*)take(W * 8);
  int64_t* d_wend = (int64_t*)take(W * 8);
  int32_t* d_wstart = (int32_t*)take((n_sys + 1) * 4);
  a.pap = (double*)take(W * kParts * 8);
  a.rrp = (double*)take(W * kParts * 8);
  a.rzp = (double*)take(W * kParts * 8);
  a.w_seg = d_wseg, a.w_beg = d_wbeg, a.w_end = d_wend, a.w_start = d_wstart;
  GS_CUDA(cudaMemcpyAsync(d_wseg, w_seg.data(), W * 4, cudaMemcpyHostToDevice, st));
  GS_CUDA(cudaMemcpyAsync(d_wbeg, w_beg.data(), W * 8, cudaMemcpyHostToDevice, st));
  GS_CUDA(cudaMemcpyAsync(d_wend, w_end.data(), W * 8, cudaMemcpyHostToDevice, st));
  GS_CUDA(cudaMemcpyAsync(d_wstart, w_start.data(), (n_sys + 1) * 4, cudaMemcpyHostToDevice, st));
  GS_CUDA(cudaMemsetAsync(h, 0, sizeof(Head), st));
  GS_TRY(ensure_row_order(ctx, mat));
  double *rl, *zl;
  GS_TRY(mas_level_vectors(ctx, mas, 1, &rl, &zl));
  const double tol2 = tol * tol;
  const dim3 g(W, kParts);
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_binit<<<g, kT, 0, st>>>(b, x, r, a); }
  GS_TRY(mas_apply_launch(ctx, mas, r, z, 1, rl, zl));
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_bdot<true><<<g, kT, 0, st>>>(r, z, p, h, a, a.rzp); }
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_bfirst<<<n_sys, 32, 0, st>>>(h, a); }
  { GS_PROF(ctx, GS_K_PCG_VECTOR); k_bfirst_running<<<1, 1, 0, st>>>(h); }

  // One PCG iteration on the context's current stream (the capture stream
  // while a graph body is being recorded).
  const bool products = mas_dot_usable(ctx, mas, 1);
  const dim3 t(kT);
  auto iteration = [&]() -> int {
    GS_TRY(spmv_launch_skip(ctx, mat, p, Ap, 1, GS_SPMV_ROW, &h->all_conv));
    auto vector = [&](auto kernel, auto... args) -> int {
      GS_PROF(ctx, GS_K_PCG_VECTOR);
      GS_CUDA(launch_chained(ctx, mat->n, kernel, g, t, 0, args...));
      return GS_OK;
    };
    GS_TRY(vector(k_bdot<false>, p, Ap, (double*)nullptr, h, a, a.pap));
    GS_TRY(vector(k_bupdate_xr, x, r, p, Ap, h, a));
    if (products) {
      GS_TRY(mas_restrict(ctx, mas, r, 1, rl, &h->all_conv));
      GS_TRY(mas_products(ctx, mas, r, z, 1, rl, zl, &h->all_conv, nullptr));
    } else {
      GS_TRY(mas_apply_launch(ctx, mas, r, z, 1, rl, zl));
    }
    GS_TRY(vector(k_bdot<false>, r, z, (double*)nullptr, h, a, a.rzp));
    GS_TRY(vector(k_bupdate_p, p, z, h, a, tol2));
    return GS_OK;
  };

  if (use_graph && max_iter > 0) {
    // One graph: a WHILE node whose body is one iteration plus the condition
    // update.  Capture needs a stream other than the legacy default stream,
    // so the body is captured on the context's private capture stream.
    if (!ctx->capture_stream) GS_CUDA(cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking));
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int status = GS_OK;
    const bool prof = ctx->prof.on;
    const cudaStream_t main_stream = ctx->stream;
    ctx->prof.on = false;  // no event records inside the captured body
    do {
      if (cudaGraphCreate(&graph, 0) != cudaSuccess) { status = GS_ERR_CUDA; break; }
      cudaGraphConditionalHandle cond;
      if (cudaGraphConditionalHandleCreate(&cond, graph, 1, cudaGraphCondAssignDefault) != cudaSuccess) {
        status = GS_ERR_CUDA;
        break;
      }
      cudaGraphNodeParams np = {};
      np.type = cudaGraphNodeTypeConditional;
      np.conditional.handle = cond;
      np.conditional.type = cudaGraphCondTypeWhile;
      np.conditional.size = 1;
      cudaGraphNode_t node;
      if (cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &np) != cudaSuccess) { status = GS_ERR_CUDA; break; }
      cudaGraph_t body = np.conditional.phGraph_out[0];
      ctx->stream = ctx->capture_stream;
      if (cudaStreamBeginCaptureToGraph(ctx->stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal) !=
          cudaSuccess) {
        status = GS_ERR_CUDA;
        break;
      }
      const cudaStream_t cs = ctx->stream;
      int s1 = iteration();
      batch::k_loop_condition<<<1, 1, 0, cs>>>(cond, h, max_iter);
      cudaError_t el = cudaGetLastError();
      cudaGraph_t captured = nullptr;
      cudaError_t ec = cudaStreamEndCapture(cs, &captured);
      if (ec == cudaSuccess && el != cudaSuccess) ec = el;
      ctx->stream = main_stream;
      if (s1 != GS_OK || ec != cudaSuccess) { status = s1 != GS_OK ? s1 : GS_ERR_CUDA; break; }
      if (cudaGraphInstantiate(&exec, graph, 0) != cudaSuccess) { status = GS_ERR_CUDA; break; }
      if (cudaGraphLaunch(exec, main_stream) != cudaSuccess) { status = GS_ERR_CUDA; break; }
    } while (false);
    ctx->stream = main_stream;
    ctx->prof.on = prof;
    if (status != GS_OK) {
      cudaGetLastError();
      set_error("gs_pcg_solve_batch: graph construction or launch failed");
    }
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (status != GS_OK) return status;
  } else {
    int* hflag = ctx->h_pinned + 256;
    for (int it = 0; it < max_iter; ++it) {
      GS_TRY(iteration());
      if ((it + 1) % 8 == 0) {
        GS_CUDA(cudaMemcpyAsync(hflag, &h->all_conv, 4, cudaMemcpyDeviceToHost, st));
        GS_CUDA(cudaStreamSynchronize(st));
        if (*hflag) break;
      }
    }
  }
  GS_CUDA(cudaGetLastError());
  std::vector<int> hconv(n_sys), hit(n_sys);
  std::vector<double> hbn(n_sys), hrr(n_sys);
  Head hh;
  GS_CUDA(cudaMemcpyAsync(hconv.data(), a.conv, n_sys * 4, cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaMemcpyAsync(hit.data(), a.iters, n_sys * 4, cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaMemcpyAsync(hbn.data(), a.bnorm2, n_sys * 8, cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaMemcpyAsync(hrr.data(), a.rr, n_sys * 8, cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaMemcpyAsync(&hh, h, sizeof(Head), cudaMemcpyDeviceToHost, st));
  GS_CUDA(cudaStreamSynchronize(st));
  bool all = true;
  for (int s = 0; s < n_sys; ++s) {
    if (iters) iters[s] = hit[s];
    if (rel_res) rel_res[s] = hbn[s] > 0 ? std::sqrt(hrr[s] / hbn[s]) : 0.0;
    all = all && hconv[s];
  }
  int flags = 0;
  GS_TRY(ctx->take_flags(&flags));
  if (hh.flags) return status_from_flags(hh.flags);
  if (flags) return status_from_flags(flags);
  if (!all) {
    set_error("gs_pcg_solve_batch: not every system converged in %d iterations", max_iter);
    return GS_ERR_MAXITER;
  }
  return GS_OK;
}

}  // namespace gs
