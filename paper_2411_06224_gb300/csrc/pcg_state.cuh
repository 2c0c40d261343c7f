// Scalars of the PCG recurrences on the device and their reductions, shared by
// the PCG kernels (pcg.cu, pcg_fused.cu) and the MAS products that take r . z
// as they write z.
#pragma once

#include "common.cuh"
#include "ff.cuh"
#include "primitives.cuh"

namespace gs {

constexpr int kMaxRhs = 32;
constexpr int kMaxRedBlocks = 1024;  // reduction blocks per right-hand side

struct PcgScalars {
  double bnorm2[kMaxRhs];
  double rz[2][kMaxRhs];  // r . z by the iteration's parity
  double rr[kMaxRhs];
  int conv[kMaxRhs];
  int bad[kMaxRhs];   // p . Ap <= 0 or a non-finite sum: stops at the end of the iteration
  int iters[kMaxRhs];
  // float-float SpMV operand (GS_SPMV_ROW_FF): |z| < 2^fz, |p| < 2^fp of the
  // iteration's parity, and the split copy of p holds p 2^(k_node - K - fsplit).
  // The other parity's fp gathers the next maximum by integer atomics.
  int fz[kMaxRhs];
  int fp[2][kMaxRhs];
  int fsplit[kMaxRhs];
  int running;        // right-hand sides that have not converged
  int all_conv;       // running == 0: kernels return at once
  int flags;
};

// Sums over the warp of kR values: afterwards every lane holds the sum of value
// sum_index<kR>(lane).  kR - 1 + 5 - log2(kR) additions instead of 5 kR.
template <int kR>
__device__ __forceinline__ int sum_index(int lane) {
  int k = 0;
#pragma unroll
  for (int h = kR / 2, o = 1; h >= 1; h /= 2, o *= 2) k += (lane & o) ? h : 0;
  return k;
}
template <int kR>
__device__ __forceinline__ double warp_sums(double (&v)[kR], int lane) {
  int o = 1;
#pragma unroll
  for (int h = kR / 2; h >= 1; h /= 2, o *= 2) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const double send = up ? v[i] : v[i + h];
      v[i] = (up ? v[i + h] : v[i]) + __shfl_xor_sync(kFull, send, o);
    }
  }
  double t = v[0];
#pragma unroll
  for (int q = kR; q < 32; q *= 2) t += __shfl_xor_sync(kFull, t, q);
  return t;
}

// Partial sums of a reduction: entry g of right-hand side k at
// sum[k * pitch + g], n of them; ex (may be null) exponent bounds alike.
struct Partials {
  double* sum = nullptr;
  int* ex = nullptr;
  int n = 0;
  int pitch = 0;
};

// Sum of one right-hand side's partials by a warp, in a fixed order: the kernel
// that needs a scalar adds the partials of the kernel before it in each of its
// blocks, so no reduction has a tail of one block.  One warp, because an FP64
// addition costs its pipe the same for one lane as for 32: all eight warps of
// each block adding took longer than the vectors themselves (65 against 41 us
// for k_pcg_p at 64^3, 8 RHS).  Every lane returns the sum.
__device__ __forceinline__ double warp_sum_partials(const Partials& a, int k) {
  const double* p = a.sum + (size_t)k * a.pitch;
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int g0 = 0; g0 < a.n; g0 += 32 * 16) {
    double q[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
      const int g = g0 + 32 * u + lane;
      q[u] = g < a.n ? __ldcg(p + g) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (g0 + 32 * u < a.n) v += q[u];  // whole warp
  }
  return warp_sum(v);
}

// alpha = rz / (p . Ap), 0 for a RHS that has stopped or whose p . Ap is not
// positive; `record` (one thread of the grid) notes the latter.
__device__ __forceinline__ double take_alpha(PcgScalars* s, int k, double pap, int parity, bool record) {
  if (s->conv[k] || s->bad[k]) return 0.0;
  const bool ok = pap > 0.0 && isfinite(pap);
  if (!ok && record) {
    atomicOr(&s->flags, isfinite(pap) ? kErrNotSPD : kErrNonFinite);
    s->bad[k] = 1;
  }
  return ok ? s->rz[parity][k] / pap : 0.0;
}

// The convergence test of RHS k after an iteration with residual norm rr:
// true if it stops (or had stopped).  `record` (one thread of the grid) keeps
// the iteration's results; others may read conv before or after, the answer is
// the same.
__device__ __forceinline__ bool test_convergence(PcgScalars* s, int k, double rr, double tol2, bool record) {
  const bool was = s->conv[k] != 0, bad = s->bad[k] != 0 || !isfinite(rr);
  const bool stop = was || bad || rr <= tol2 * s->bnorm2[k];
  if (record && !was) {
    if (!isfinite(rr))
      atomicOr(&s->flags, kErrNonFinite);
    else if (!bad) {
      s->rr[k] = rr;
      s->iters[k] += 1;
    }
    if (stop) {
      s->conv[k] = 1;
      if (atomicSub(&s->running, 1) == 1) s->all_conv = 1;
    }
  }
  return stop;
}

// Programmatic dependent launch: a kernel may be resident before the one ahead
// of it in the stream has finished; it waits here for that kernel's results.
// Without the launch attribute both are no-ops.  Such a kernel lives while the one
// before it writes, so its pointers to the iteration's vectors and words are not
// `const __restrict__`: that would say nobody writes them meanwhile, and let the
// compiler load them ahead of the wait or without coherence.  Tables older than
// the solve are.
__device__ __forceinline__ void wait_for_previous_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_kernel_launch() { asm volatile("griddepcontrol.launch_dependents;"); }

// Up to this many block rows x right-hand sides an iteration is bound by its
// launches and latencies, beyond it by bytes and arithmetic.  Kernels of the
// first kind are chained (below) and fused further (pcg.cu).  24 iterations, float-
// float product, with / without, by rows x RHS, FP64 preconditioner: 182,000 (45^3 x
// 2) 3.25 / 4.21 ms; 375,000 (50^3 x 3) 5.19 / 5.59; 547,000 (45^3 x 6) 5.52 / 6.07;
// 702,000 (56^3 x 4) 6.98 / 7.27; 750,000 (50^3 x 6) 7.21 / 7.63; 786,000 (64^3 x 3)
// 9.35 / 9.13; 1.05M (64^3 x 4) 9.55 / 9.26; 2.1M (64^3 x 8) 14.4 / 12.9.  FP32: 702,000
// 5.60 / 6.18; 1.05M 7.63 / 7.71; 1.4M (56^3 x 8) 9.59 / 9.22.
constexpr int64_t kSmallWork = 750 << 10;

// Launch `kernel` on the context's stream so that, for small work, its blocks
// may become resident while the kernel before it drains (the kernel calls
// wait_for_previous_kernel); larger kernels run by themselves: waiting blocks
// take room from the blocks still to come.
template <typename... P, typename... A>
inline cudaError_t launch_chained(gs_ctx ctx, int64_t work, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                  A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = ctx->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = work <= kSmallWork ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace gs
