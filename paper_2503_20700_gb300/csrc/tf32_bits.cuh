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

}  // namespace dmrg
