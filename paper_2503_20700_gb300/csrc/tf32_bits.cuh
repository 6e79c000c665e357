// float64 from float32, and the TF32 parts of a float64, without the float64
// pipe: GB300 converts two numbers a clock and SM on it, which bound the operand
// split and the chunk reduction of the tcgen05 contraction.  Ordinary numbers go
// by integer operations, with the values that the conversions give, the rest by
// the conversions.  Compiles for the host too (for tests).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace dmrg {

__host__ __device__ __forceinline__ uint32_t float_bits(float x) {
  uint32_t u;
  memcpy(&u, &x, 4);
  return u;
}
__host__ __device__ __forceinline__ float bits_float(uint32_t u) {
  float x;
  memcpy(&x, &u, 4);
  return x;
}

// TF32 (11 bits), to nearest, ties away from zero
__host__ __device__ __forceinline__ uint32_t tf32_round(float x) {
#ifdef __CUDA_ARCH__
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
#else
  const uint32_t u = float_bits(x);
  return ((u >> 23) & 0xFFu) == 0xFFu ? u : (u + 0x1000u) & ~0x1FFFu;
#endif
}

__host__ __device__ __forceinline__ double widen(float x) {
  const uint32_t u = float_bits(x), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u >= 0x7F000000u && m != 0u) return (double)x;  // subnormal, infinite, NaN
  const uint64_t d = (uint64_t)((u & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u)) << 32 | (uint32_t)(u << 29);
  double r;
  memcpy(&r, &d, 8);
  return r;
}

// hi = tf32(float(v)), lo = tf32(float(v - hi))
__host__ __device__ __forceinline__ void split_tf32(double v, float& hi, float& lo) {
  uint64_t bits;
  memcpy(&bits, &v, 8);
  const uint32_t vh = (uint32_t)(bits >> 32), vl = (uint32_t)bits;
  const uint32_t be = (vh >> 20) & 0x7FFu, sign = vh & 0x80000000u;
  if (be - 949u > 200u) {  // not in 2^-74 ... 2^127
    if ((vh << 1 | vl) == 0u) {
      hi = bits_float(vh);
      lo = 0.0f;
      return;
    }
    hi = bits_float(tf32_round((float)v));
    lo = bits_float(tf32_round((float)(v - (double)hi)));
    return;
  }
  // |v| to nearest even in 24 bits (a carry goes into the exponent), then to
  // 11 bits
  const uint32_t m23 = (vh & 0xFFFFFu) << 3 | vl >> 29, rest = vl & 0x1FFFFFFFu, half = 1u << 28;
  const uint32_t f = ((be - 896u) << 23 | m23) + ((rest > half || (rest == half && (m23 & 1u))) ? 1u : 0u);
  const uint32_t h = tf32_round(bits_float(f));
  // |v| - hi in units of 2^(be - 1075), at most 2^42
  const long long M = (long long)((vh & 0xFFFFFu) | 0x100000u) << 32 | vl;
  const long long H = (long long)((h & 0x7FFFFFu) | 0x800000u) << (29 + (int)((h >> 23) + 896u - be));
  const long long D = M - H;
  // to 24 bits: whole if it fits into 32, else 26 to 31 bits of it, the others
  // leaving their trace in the last one for the rounding
  const bool wide = D >= (1ll << 37) || D < -(1ll << 37);
  const int drop = D == (long long)(int)D ? 0 : wide ? 12 : 6;
  const int t = (int)(D >> drop) | (int)((D & ((1 << drop) - 1)) != 0);
  const float l = (float)t * bits_float((be - 948u + (uint32_t)drop) << 23);
  hi = bits_float(h | sign);
  lo = bits_float(tf32_round(sign ? -l : l));
}

__host__ __device__ __forceinline__ int leading_zeros(uint64_t x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

// (double)x + (double)y of a pair whose second part is the smaller
__host__ __device__ __forceinline__ double pair_sum(float x, float y) {
  const uint32_t ux = float_bits(x), uy = float_bits(y), ex = (ux >> 23) & 0xFFu, ey = (uy >> 23) & 0xFFu;
  if ((uy << 1) == 0u) return widen(x);
  // both ordinary, the second at least one binary place down
  if (ex - 1u >= 254u || ey - 1u >= 254u || ey >= ex) return widen(x) + widen(y);
  const uint32_t d = ex - ey;
  const uint64_t mx = (uint64_t)((ux & 0x7FFFFFu) | 0x800000u) << 39;  // leading one at bit 62
  uint64_t my = (uint64_t)((uy & 0x7FFFFFu) | 0x800000u) << 39;
  // what is shifted out leaves its trace in the last bit
  my = d < 63u ? (my >> d) | (uint64_t)((my & ((1ull << d) - 1)) != 0) : 1u;
  const uint64_t s = ((ux ^ uy) >> 31) ? mx - my : mx + my;
  const int n = leading_zeros(s);  // 0 ... 2
  const uint64_t top = s << n, q = top >> 11;
  const uint32_t rest = (uint32_t)top & 0x7FFu;
  const uint64_t up = rest > 0x400u || (rest == 0x400u && (q & 1u));
  const uint64_t b = (((uint64_t)(ex + 896u - (uint32_t)n) << 52) + q + up) | (uint64_t)(ux >> 31) << 63;
  double r;
  memcpy(&r, &b, 8);
  return r;
}

}  // namespace dmrg
