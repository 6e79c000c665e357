// Host check of tf32_bits.cuh: the integer conversions against the conversions
// themselves, bit by bit (but for the sign of a zero remainder), over exponents
// at and beyond their range, mantissas with runs of zeros and ones, ties.
#include <cmath>
#include <cstdio>
#include <random>

#include "tf32_bits.cuh"

using namespace dmrg;

static long bad = 0;
static double from(uint64_t u) {
  double x;
  memcpy(&x, &u, 8);
  return x;
}
static uint64_t of(double x) {
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
}
static void check(double v) {
  float h, l;
  split_tf32(v, h, l);
  const float h0 = bits_float(tf32_round((float)v)), l0 = bits_float(tf32_round((float)(v - (double)h0)));
  if (float_bits(h) != float_bits(h0) || (float_bits(l) != float_bits(l0) && !(l == 0.0f && l0 == 0.0f)))
    if (++bad < 10) std::printf("%a: %a %a, not %a %a\n", v, h, l, h0, l0);
}

int main() {
  std::mt19937_64 r(1);
  const uint64_t mant = 0xFFFFFFFFFFFFFull;
  for (long i = 0; i < 4000000; ++i) {
    const uint64_t b = r(), sign = b & 0x8000000000000000ull, cut = (1ull << (r() % 53)) - 1;
    uint64_t e = 940 + (b >> 40) % 220, m = r() & mant;
    if (i % 5 == 0) e = (b >> 40) % 1150;
    if (i % 5 == 1) m &= ~cut;
    if (i % 5 == 2) m |= cut;
    if (i % 5 == 3) m = (m >> 29 << 29) | (1ull << 28);
    check(from(sign | e << 52 | m));
    const float x = bits_float((uint32_t)r());
    if (!std::isnan(x) && of(widen(x)) != of((double)x)) ++bad;
  }
  for (uint64_t e = 0; e < 1151; ++e)
    for (uint64_t m : {uint64_t(0), mant, uint64_t(1), mant - 1, uint64_t(1) << 41, uint64_t(1) << 42, uint64_t(1) << 28})
      check(from(e << 52 | m));
  for (float x : {0.0f, -0.0f, 1.17549435e-38f, 3.4028234e38f, -1e-40f, INFINITY, -INFINITY})
    if (of(widen(x)) != of((double)x)) ++bad;
  for (long i = 0; i < 8000000; ++i) {
    const uint64_t b = r();
    const float x = bits_float((uint32_t)b);
    uint32_t u = (uint32_t)(b >> 32);
    // most of them near below x
    if (i % 4) {
      const uint32_t ex = (float_bits(x) >> 23) & 0xFFu, dn = (uint32_t)(r() % 70);
      u = (u & 0x807FFFFFu) | (ex > dn ? ex - dn : 0u) << 23;
      if (i % 4 == 1) u &= ~0u << (r() % 24);
    }
    const float y = bits_float(u);
    if (std::isnan(x) || std::isnan(y) || std::isinf(x) || std::isinf(y)) continue;
    if (of(pair_sum(x, y)) != of((double)x + (double)y) && ++bad < 20)
      std::printf("%a + %a: %a, not %a\n", x, y, pair_sum(x, y), (double)x + (double)y);
  }
  if (bad) return 1;
  std::printf("conversions agree\n");
  return 0;
}
