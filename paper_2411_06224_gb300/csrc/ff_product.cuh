// Float-float product of a 3x3 block (or its transpose) with the split operand
// of up to kR right-hand sides, and its accumulators: the arithmetic of
// spmv_ff.cu, shared with PCG's own product (pcg_fused.cu).
#pragma once

#include "ff.cuh"
#include "primitives.cuh"

namespace gs {

// Accumulate the term (ah + al)(xh + xl) into the pair (S, L).  The rounded
// intrinsics keep the compiler from contracting or reordering the
// transformations.  The term's small parts are added among themselves first, so
// that only one of the four roundings is at the size of L.
__device__ __forceinline__ void ff_term(float ah, float al, float xh, float xl, float& S, float& L) {
  const float p = __fmul_rn(ah, xh);
  const float e = __fmaf_rn(ah, xh, -p);
  const float s = __fadd_rn(S, p);
  const float bp = __fsub_rn(s, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(s, bp)), __fsub_rn(p, bp));
  S = s;
  L = __fadd_rn(L, __fmaf_rn(al, xh, __fmaf_rn(ah, xl, __fadd_rn(err, e))));
}

// (S, L) += (S2, L2): two-sum of the large parts, the rest gathered in L.
__device__ __forceinline__ void ff_merge(float& S, float& L, float S2, float L2) {
  const float s = __fadd_rn(S, S2);
  const float bp = __fsub_rn(s, S);
  const float err = __fadd_rn(__fsub_rn(S, __fsub_rn(s, bp)), __fsub_rn(S2, bp));
  S = s;
  L = __fadd_rn(L, __fadd_rn(L2, err));
}

// f * 2^e as a double, built from f's bit pattern (no conversion
// instruction; on this part conversions run on the FP64 pipe).  A zero or
// subnormal f gives 0; e keeps the result inside the double range here.
__device__ __forceinline__ double f32_times_pow2(float f, int e) {
  const unsigned b = __float_as_uint(f);
  const int fe = (int)((b >> 23) & 0xffu);
  if (fe == 0) return 0.0;
  const int de = min(max(fe - 127 + 1023 + e, 1), 2046);
  const unsigned hi = (b & 0x80000000u) | ((unsigned)de << 20) | ((b & 0x7fffffu) >> 3);
  return __hiloint2double((int)hi, (int)(b << 29));
}

template <int kV>
struct FFSum {
  float S[kV], L[kV];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int q = 0; q < kV; ++q) S[q] = 0.f, L[q] = 0.f;
  }
  // (S, L) = two_sum(S, L): the same sum, L small again.
  __device__ __forceinline__ void settle() {
#pragma unroll
    for (int q = 0; q < kV; ++q) {
      const float s = __fadd_rn(S[q], L[q]);
      const float bp = __fsub_rn(s, S[q]);
      L[q] = __fadd_rn(__fsub_rn(S[q], __fsub_rn(s, bp)), __fsub_rn(L[q], bp));
      S[q] = s;
    }
  }
  // Sum over kLanes neighbouring lanes, in a fixed order.
  template <int kLanes>
  __device__ __forceinline__ void merge() {
#pragma unroll
    for (int q = 0; q < kV; ++q) {
#pragma unroll
      for (int o = kLanes / 2; o > 0; o >>= 1) {
        const float S2 = __shfl_xor_sync(kFull, S[q], o, kLanes);
        const float L2 = __shfl_xor_sync(kFull, L[q], o, kLanes);
        ff_merge(S[q], L[q], S2, L2);
      }
    }
  }
  __device__ __forceinline__ double value(int q, int e) const {
    return f32_times_pow2(S[q], e) + f32_times_pow2(L[q], e);
  }
};

// acc += H x for right-hand sides 0 .. nh - 1 of the column operand xb (3 pairs
// each); vec: xb is 16-byte aligned, two RHS at a time.
template <int kR>
__device__ __forceinline__ void ff_block_product(const float2 (&H)[9], const float2* xb, int nh, bool vec,
                                                 FFSum<kR * 3>& acc) {
#pragma unroll
  for (int q = 0; q < kR; q += 2) {
    float2 xv[6];
    if (vec) {
      if (q < nh) {
        const float4* x4 = reinterpret_cast<const float4*>(xb + 3 * q);
        const float4 a = x4[0], b = x4[1], c = x4[2];
        xv[0] = make_float2(a.x, a.y), xv[1] = make_float2(a.z, a.w), xv[2] = make_float2(b.x, b.y);
        xv[3] = make_float2(b.z, b.w), xv[4] = make_float2(c.x, c.y), xv[5] = make_float2(c.z, c.w);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 6; ++i)
        if (q + i / 3 < nh && (q + i / 3) < kR) xv[i] = xb[3 * q + i];
    }
#pragma unroll
    for (int qq = 0; qq < 2; ++qq) {
      const int qi = q + qq;
      if (qi < kR && qi < nh) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
#pragma unroll
          for (int j = 0; j < 3; ++j)
            ff_term(H[3 * c + j].x, H[3 * c + j].y, xv[3 * qq + j].x, xv[3 * qq + j].y, acc.S[3 * qi + c],
                    acc.L[3 * qi + c]);
        }
      }
    }
  }
}

}  // namespace gs
