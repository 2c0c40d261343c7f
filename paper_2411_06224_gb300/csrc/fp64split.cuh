// Integer helpers of the FP64-accurate tensor-core products: exponent
// fields, exact scaling of a double to an integer and the rounding of a
// wide integer times a power of two back to a double.  Every step runs on
// the integer units, so no FP64 instruction is spent on the splits.
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace gs {

// Biased exponent field of a double (0 for zero / subnormal).
__device__ __forceinline__ int biased_exp(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// rint(v * 2^(56 - b)) for |v| < 2^(b-1), in integer arithmetic (round half
// to even) without branches, so |result| <= 2^55; 0 for zeros and subnormals.
__device__ __forceinline__ long long scaled_rint(double v, int b) {
  const long long bits = __double_as_longlong(v);
  const int eb = (int)((bits >> 52) & 0x7FF);
  // value = mant 2^(eb - 1075); times 2^(56 - b) = (4 mant) 2^-s, s >= 0 by the bound on |v|
  const unsigned long long x4 = eb ? ((unsigned long long)bits & 0xFFFFFFFFFFFFFull | 0x10000000000000ull) << 2 : 0ull;
  const int s = min(max(1021 - eb + b, 0), 60);  // beyond 57 everything rounds to 0
  const unsigned long long half = (1ull << s) >> 1;
  const unsigned long long up = half ? half - 1 + ((x4 >> s) & 1) : 0ull;
  const long long q = (long long)((x4 + up) >> s);
  return bits < 0 ? -q : q;
}

// Balanced digits of y (|y| < 2^55) are the plain digits of y + C minus the
// offset, C holding the offset in every digit (base 256) or every digit but the
// top one (base 128), so each digit is one bit-field extract.

// The BF16 of a small integer is the top half of the float 1.5 2^23 + d - 1.5
// 2^23 (exact: d has at most 8 significant bits).
__device__ __forceinline__ uint16_t small_int_bf16_bits(int d) {
  return (uint16_t)(__float_as_uint(__int_as_float(0x4B400000 + d) - 12582912.0f) >> 16);
}

// Base 256, digits 0..6 (the most significant first; d_0 in [-128, 128], the
// others in [-128, 127]) as F16, written at 0 .. 6 * 128 of col; an eighth, zero digit at 7 * 128.  With 128
// added to every digit they are the bytes of one integer, and 1024 + u, u <= 256,
// is the F16 with the bits 0x6400 + u.
constexpr unsigned long long kBias256 = 0x80808080808080ull;
__device__ __forceinline__ void write_digits256_f16(long long y, unsigned char* col) {
  const unsigned long long z = (unsigned long long)y + kBias256;
  const uint32_t lo = (uint32_t)z, hi = (uint32_t)(z >> 32);  // hi < 2^25
  const uint32_t u[7] = {hi >> 16, (hi >> 8) & 255u, hi & 255u, lo >> 24, (lo >> 16) & 255u, (lo >> 8) & 255u, lo & 255u};
  const __half off = __ushort_as_half(0x6480);  // 1024 + 128
#pragma unroll
  for (int p = 0; p < 7; ++p)
    *(uint16_t*)(col + p * 128) = __half_as_ushort(__hsub(__ushort_as_half((unsigned short)(0x6400u + u[p])), off));
  *(uint16_t*)(col + 7 * 128) = 0;
}

// Byte p (0: the most significant of 7) of four integers as one word, z0's lowest.
__device__ __forceinline__ void bytes_of_four(const unsigned long long (&z)[4], uint32_t (&w)[7]) {
  const uint32_t l0 = (uint32_t)z[0], l1 = (uint32_t)z[1], l2 = (uint32_t)z[2], l3 = (uint32_t)z[3];
  const uint32_t h0 = (uint32_t)(z[0] >> 32), h1 = (uint32_t)(z[1] >> 32), h2 = (uint32_t)(z[2] >> 32),
                 h3 = (uint32_t)(z[3] >> 32);
  const uint32_t a = __byte_perm(l0, l1, 0x5140), b = __byte_perm(l2, l3, 0x5140);  // bytes 0, 0', 1, 1'
  const uint32_t c = __byte_perm(l0, l1, 0x7362), d = __byte_perm(l2, l3, 0x7362);  // bytes 2, 2', 3, 3'
  const uint32_t e = __byte_perm(h0, h1, 0x5140), f = __byte_perm(h2, h3, 0x5140);
  w[6] = __byte_perm(a, b, 0x5410), w[5] = __byte_perm(a, b, 0x7632);
  w[4] = __byte_perm(c, d, 0x5410), w[3] = __byte_perm(c, d, 0x7632);
  w[2] = __byte_perm(e, f, 0x5410), w[1] = __byte_perm(e, f, 0x7632);
  w[0] = __byte_perm(__byte_perm(h0, h1, 0x0062), __byte_perm(h2, h3, 0x0062), 0x5410);
}

// Four digit bytes (digit + 128 each) as two F16 pairs.
__device__ __forceinline__ void expand_digit_bytes(uint32_t w, uint32_t& d01, uint32_t& d23) {
  const uint32_t off = 0x64806480u;
  const uint32_t a = __byte_perm(w, 0x64646464u, 0x4140), b = __byte_perm(w, 0x64646464u, 0x4342);
  const __half2 o = *reinterpret_cast<const __half2*>(&off);
  const __half2 x = __hsub2(*reinterpret_cast<const __half2*>(&a), o), y = __hsub2(*reinterpret_cast<const __half2*>(&b), o);
  d01 = *reinterpret_cast<const uint32_t*>(&x);
  d23 = *reinterpret_cast<const uint32_t*>(&y);
}

// base 128, digits 0..7 (d_0 in [-64, 64], the others in [-64, 63]) into d[]
__device__ __forceinline__ void digits128_fast(long long y, int (&d)[8]) {
  const long long z = y + 0x1020408102040LL;  // 64 in digits 1..7: 64 (128^7 - 1) / 127
  const uint32_t lo = (uint32_t)z, hi = (uint32_t)((unsigned long long)z >> 32);
  d[0] = (int)(z >> 49);
  d[1] = (int)((hi >> 10) & 127u) - 64;
  d[2] = (int)((hi >> 3) & 127u) - 64;
  d[3] = (int)(((hi << 4) | (lo >> 28)) & 127u) - 64;
  d[4] = (int)((lo >> 21) & 127u) - 64;
  d[5] = (int)((lo >> 14) & 127u) - 64;
  d[6] = (int)((lo >> 7) & 127u) - 64;
  d[7] = (int)(lo & 127u) - 64;
}

// (hi 2^S + lo) 2^e as the nearest double (ties to even), |hi|, |lo| < 2^52,
// 24 <= S <= 40, in 64-bit integer arithmetic: the 128-bit sum as two words,
// its magnitude normalised to a leading one in bit 63 of `top`, the bits
// below it OR-ed into a sticky word.  Results below the normal range flush
// to zero.
__host__ __device__ __forceinline__ int clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

__host__ __device__ __forceinline__ double combine_to_double(long long hi, long long lo, int S, int e) {
  unsigned long long L0 = (unsigned long long)hi << S;
  long long H = hi >> (64 - S);  // sign-extended high word of hi 2^S
  unsigned long long L = L0 + (unsigned long long)lo;
  H += (lo < 0 ? -1 : 0) + (L < L0 ? 1 : 0);
  unsigned long long sign = 0;
  if (H < 0) {  // magnitude of the 128-bit two's complement value
    sign = 0x8000000000000000ULL;
    L = ~L + 1;
    H = ~H + (L == 0 ? 1 : 0);
  }
  const unsigned long long UH = (unsigned long long)H;
  if (UH == 0 && L == 0) return 0.0;
  int lz;
  unsigned long long top, sticky;
  if (UH) {
    lz = clz64(UH);  // >= 1: |hi 2^S + lo| < 2^127
    top = (UH << lz) | (L >> (64 - lz));
    sticky = L << lz;
  } else {
    const int l = clz64(L);
    lz = 64 + l;
    top = L << l;
    sticky = 0;
  }
  unsigned long long m = top >> 11;  // 53 bits, leading one at bit 52
  const unsigned long long g = top & 0x7FFULL;
  int E = 127 - lz + e;  // value = 1.f 2^E
  if (g > 0x400ULL || (g == 0x400ULL && (sticky != 0 || (m & 1ULL)))) {
    if (++m == (1ULL << 53)) {
      m >>= 1;
      ++E;
    }
  }
  if (E < -1022) return 0.0;
  const unsigned long long bits = sign | ((unsigned long long)(E + 1023) << 52) | (m & 0xFFFFFFFFFFFFFULL);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double v;
  __builtin_memcpy(&v, &bits, 8);
  return v;
#endif
}

}  // namespace gs
