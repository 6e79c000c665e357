// Float64 grouped GEMM by exact digit products on tcgen05 (gemm_digits.cuh).
//
// gemm_digits_kernel is persistent (one CTA per SM, tasks dealt longest
// first).  A k-step of 16 brings the nine digits of 128 rows of op(A) and 64
// columns of op(B) (54 KB, 18 bulk copies) into one of three stages; digit i
// of A meets the digits 0..7-i of B, stacked along N, so one MMA of N = 256
// covers four digits of B and its output columns are the accumulators
// i..i+3; digit 8-i of B comes on top of the last accumulator by an MMA of its
// own (N = 64).  21 MMAs a k-step.  The eight accumulators (128 x 64 FP32 each)
// fill TMEM.
//
// What bounds it: shared memory for long segments (a k-step's MMAs read 174 KB
// and its copies write 54 KB), the float64 pipe for short ones (three operations
// per output and segment at two a clock and SM, 12300 clocks a tile).  The tile
// is 128 x 64 because eight accumulators of that size are all of TMEM; N = 64
// alone would read shared memory at 48 clocks per 32-clock MMA, which the
// stacked form avoids.  Measured, 152 tiles at once: 1.17 us a k-step (0.96 with
// eight digits and 12 MMAs).  601 products of 200 x 200 x 200 (the rotation of
// 600 Cholesky vectors): 0.6 ms (0.46) and 0.18 ms for the split (0.16), 12
// TFLOP/s of float64; the FMA kernel needs 13 ms (0.74 TFLOP/s, 1.25 nominal
// peak).
#include <algorithm>
#include <stdexcept>
#include <string>

#include "gemm_digits.cuh"
#include "kattr.hpp"

namespace dmrg {

namespace {

constexpr int NSTAGE = 3;
constexpr int A_SLICE = 16 * kDigUnit, B_SLICE = 8 * kDigUnit;  // 128 and 64 rows of one digit
constexpr int A_BYTES = kDigSlices * A_SLICE, B_BYTES = kDigSlices * B_SLICE;
constexpr int STAGE = A_BYTES + B_BYTES;
// per epilogue warp: 16 x 32 outputs, turned from row-per-lane (TMEM) to
// column-per-lane (coalesced C)
constexpr int TURN_LD = 33;
constexpr int OFF_TURN = NSTAGE * STAGE, TURN_BYTES = 16 * TURN_LD * 8;
constexpr int SMEM_BYTES = OFF_TURN + 8 * TURN_BYTES + 1024;
constexpr int CHUNK = 16;  // k-steps of 16 between drains: 256 exact terms
constexpr int NTHREADS = 384;
constexpr unsigned long long kDrainNs = 2000000000ull;  // what a CTA that gave up waits for its own work in flight
constexpr int kExpRange = 400;

enum { B_FULL = 0, B_EMPTY = B_FULL + NSTAGE, B_SF = B_EMPTY + NSTAGE, B_SE, B_MF, B_ME = B_MF + 2,
       B_DONE = B_ME + 2, B_COUNT };

// what the epilogue needs of a segment, gathered one segment ahead by a warp
// of its own (the dependent loads task - segment - operand took a third of the
// epilogue's time)
struct Meta {
  DigTask t;
  double alpha;
  long long ua, ub;  // masks of the operands
  int sa, sb;        // their rows per 16 columns
  int k, plain;
  int ea[kDigTileM], eb[kDigTileN];  // row and column exponents
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// K-major, no swizzle: core matrices 128 B apart along k, 256 B between 8-row groups
__device__ __forceinline__ uint64_t desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | (uint64_t)(128 >> 4) << 16 | (uint64_t)(kDigUnit >> 4) << 32 |
         (uint64_t)1 << 46;
}
// kind::f16, bf16 operands, FP32 accumulator, both operands K-major, M = 128
__device__ __forceinline__ uint32_t idesc(int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kDigTileM >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc));
}
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void arrive_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// bulk copy of `bytes` (a multiple of 256, 256-byte aligned on both sides)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
__device__ __forceinline__ bool test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// wait bounded by wait_ns (0: by its first probe); false when it ran out or
// another role of the CTA gave up.  Every wait is on this CTA's own work.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, volatile int* abort,
                                         unsigned long long wait_ns) {
  if (wait_ns == 0) return test_wait(bar, parity);
  if (try_wait(bar, parity)) return true;  // before the clock is read, which takes longer than most waits
  const unsigned long long t0 = global_ns();
  for (;;) {
    if (try_wait(bar, parity)) return true;
    if (*abort || global_ns() - t0 > wait_ns) return false;
  }
}
// columns of a tile on the tensor pipe (steps of 16)
__device__ __forceinline__ int tile_width(int left) { return min(kDigTileN, (left + 15) & ~15); }
// h 2^32 + l rounded once to float64, |h| < 2^51: with the integers placed in
// the mantissas, (2^52 + 2^51 + h) - (2^52 + 2^51 + 2^20) = h - 2^20 is exact
// and the fused sum (h - 2^20) 2^32 + (2^52 + l) is the value
__device__ __forceinline__ double combined(long long h, uint32_t l) {
  const double u = __hiloint2double(0x43380000 + (int)(h >> 32), (int)(uint32_t)h) - 6755399442104320.0;
  return fma(u, 4294967296.0, __hiloint2double(0x43300000, (int)l));
}
__device__ __forceinline__ long long mad_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}
__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(addr));
}

// ---------------------------------------------------------------- operand split
__device__ __forceinline__ double elem(const DigOperand& o, int r, int c) {
  return o.trans ? __ldg(o.src + (size_t)c * o.ld + r) : __ldg(o.src + (size_t)r * o.ld + c);
}
// byte `byte` of word (digit s + 128) as the digit times 2^-8s
template <int S>
__device__ __forceinline__ float digit_float(uint32_t word, int byte) {
  // (2^23 + byte) 2^-8s, minus (2^23 + 128) 2^-8s
  constexpr uint32_t one = 0x4B000000u - ((uint32_t)S << 26);
  constexpr double weight = 1.0 / (double)(1ull << (8 * (S < 8 ? S : 7))) / (S < 8 ? 1.0 : 256.0);
  return __uint_as_float(__byte_perm(word, one, 0x7440 + byte)) - (float)(8388736.0 * weight);
}

// 32 rows of one operand per CTA: row maxima, then the digits.  Bound by the
// latency of its loads for the matrices of a sweep and by HBM and the integer
// pipe together for large ones (8 B read twice, 18 B written, some fifty
// integer operations per element), so a thread loads the eight columns of its
// row before it uses the first.  Its eight 16-byte stores, one per digit, fill
// 512 contiguous bytes each with those of its warp.
constexpr int SPLIT_THREADS = 512;
__device__ __forceinline__ void load8(const DigOperand& o, int r, int c0, double (&x)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) x[i] = (r < o.rows && c0 + i < o.k) ? elem(o, r, c0 + i) : 0.0;
}

__global__ void __launch_bounds__(SPLIT_THREADS) split_digits_kernel(const DigOperand* __restrict__ ops,
                                                                     const DigSplit* __restrict__ splits,
                                                                     unsigned char* __restrict__ pool,
                                                                     unsigned char* __restrict__ last,
                                                                     int* __restrict__ exps,
                                                                     DigMask* __restrict__ masks,
                                                                     uint16_t* __restrict__ nonzero,
                                                                     int* __restrict__ special) {
  __shared__ unsigned rowmax[32];
  constexpr int KSTEP = SPLIT_THREADS / 64;  // k-blocks of 16 in flight
  const DigSplit sp = splits[blockIdx.x];
  const DigOperand o = ops[sp.op];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gl = (warp & 1) * 2 + (lane >> 4);  // row group within the block
  const int rl = gl * 8 + (lane & 7), r = sp.r0 + rl;
  const int kc = (lane >> 3) & 1;
  const int nkb = (o.k + 15) >> 4;
  if (threadIdx.x < 32) rowmax[threadIdx.x] = 0u;
  __syncthreads();
  unsigned mx = 0u;
  for (int kb = warp >> 1; kb < nkb; kb += KSTEP) {
    double x[8];
    load8(o, r, kb * 16 + kc * 8, x);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      // high word of |x|; a subnormal with a zero high word still counts
      const unsigned hi = (unsigned)__double2hiint(x[i]) & 0x7FFFFFFFu;
      mx = max(mx, max(hi, (unsigned)(__double2loint(x[i]) != 0)));
    }
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  if (kc == 0 && mx) atomicMax(&rowmax[rl], mx);
  __syncthreads();
  const int be_row = (int)(rowmax[rl] >> 20);
  if (threadIdx.x < 32 && sp.r0 + (int)threadIdx.x < o.rows) {
    const unsigned m = rowmax[threadIdx.x];
    const int be = (int)(m >> 20);
    exps[o.eoff + sp.r0 + threadIdx.x] = m ? be - 1022 : 0;
    if (m && (be < 1023 - kExpRange || be > 1023 + kExpRange)) special[sp.op] = 1;
  }
  const int g = (sp.r0 >> 3) + gl;
  const bool stored = g < o.groups;  // rows beyond the operand inside its last group are zero
  const size_t at0 = (size_t)g * kDigUnit + kc * 128 + (lane & 7) * 16;
  unsigned char* const base = pool + (size_t)o.unit * kDigUnit + at0;
  unsigned char* const base_last = last + (size_t)o.unit / kDigSums * kDigUnit + at0;
  for (int kb = warp >> 1; kb < nkb; kb += KSTEP) {
    const int c0 = kb * 16 + kc * 8;
    double x[8];
    load8(o, r, c0, x);
    uint32_t w[kDigSlices][4];
    DigMask mk = make_uint2(0u, 0u);
    unsigned nz = 0u;
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      float f[2][kDigSlices];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(x[i + q]);
        const int be = (int)((bits >> 52) & 0x7FF);
        unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | 1ull << 52;
        // F of up to 71 bits: top 2^64 + m
        const int sh = be - be_row + 17;  // at most 17
        uint32_t top = 0u;
        if (be == 0 || sh < -54) {
          m = 0;
        } else if (sh >= 0) {
          top = sh > 11 ? (uint32_t)(m >> (64 - sh)) : 0u;
          m <<= sh;
        } else {
          m = (m + (1ull << (-sh - 1))) >> -sh;
        }
        if ((long long)bits < 0) {
          m = 0ull - m;
          top = ~top + (m == 0ull);
        }
        const unsigned long long u = m + 0x8080808080808080ull;  // every digit + 128
        top += 0x80u + (u < 0x8080808080808080ull);
        const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u;
        f[q][0] = digit_float<0>(top, 0);
        f[q][1] = digit_float<1>(uh, 3);
        f[q][2] = digit_float<2>(uh, 2);
        f[q][3] = digit_float<3>(uh, 1);
        f[q][4] = digit_float<4>(uh, 0);
        f[q][5] = digit_float<5>(ul, 3);
        f[q][6] = digit_float<6>(ul, 2);
        f[q][7] = digit_float<7>(ul, 1);
        f[q][8] = digit_float<8>(ul, 0);
        const int down = be_row - be;
        mk.x |= be && down <= 5 ? 1u << (i + q) : 0u;
        mk.x |= be && down <= 7 ? 0x10000u << (i + q) : 0u;
        mk.y |= be && down <= 2 ? 1u << (i + q) : 0u;
        mk.y |= be && down <= 10 ? 0x10000u << (i + q) : 0u;
        nz |= bits << 1 ? 1u << (i + q) : 0u;
      }
#pragma unroll
      for (int s = 0; s < kDigSlices; ++s)
        w[s][i >> 1] = __byte_perm(__float_as_uint(f[0][s]), __float_as_uint(f[1][s]), 0x7632);
    }
    if (stored) {
#pragma unroll
      for (int s = 0; s < kDigSums; ++s)
        *reinterpret_cast<uint4*>(base + ((size_t)kb * kDigSums + s) * o.groups * kDigUnit) =
            make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
      *reinterpret_cast<uint4*>(base_last + (size_t)kb * o.groups * kDigUnit) =
          make_uint4(w[kDigSums][0], w[kDigSums][1], w[kDigSums][2], w[kDigSums][3]);
    }
    // the two halves of the 16 columns
    mk.x <<= 8 * kc;
    mk.y <<= 8 * kc;
    mk.x |= __shfl_xor_sync(0xffffffffu, mk.x, 8);
    mk.y |= __shfl_xor_sync(0xffffffffu, mk.y, 8);
    nz <<= 8 * kc;
    nz |= __shfl_xor_sync(0xffffffffu, nz, 8);
    if (stored && kc == 0) {
      const size_t at = (size_t)o.unit + (size_t)kb * 8 * o.groups + r;
      masks[at] = mk;
      nonzero[at] = (uint16_t)nz;
    }
  }
}

// ---------------------------------------------------------------- products
// Bit c: the output of this lane's row and column c (of `ncol`) is to be left
// out: no term of it is known to reach 2^-14 of 2^ea 2^eb, and not all are zero.
// ma, na: this lane's row (has_row: there is one), mb, nb: column 0, at k-block 0.
// Two k-blocks at a time, for the latency of their loads; they settle a dense
// operand, and 400 integer operations of a warp stand beside 3000 clocks of the
// products of two k-blocks.
__device__ __forceinline__ uint32_t outputs_left(bool has_row, const DigMask* ma, const uint16_t* na, int sa,
                                                 const DigMask* mb, const uint16_t* nb, int sb, int nkb, int ncol) {
  uint32_t open = has_row ? 0xFFFFFFFFu >> (32 - ncol) : 0u;  // not settled yet
  for (int kb = 0; kb < nkb; kb += 2) {
    const int k1 = min(kb + 1, nkb - 1);
    const uint2 z = make_uint2(0u, 0u);
    const uint2 a0 = has_row ? __ldg(ma + (size_t)kb * sa) : z, a1 = has_row ? __ldg(ma + (size_t)k1 * sa) : z;
    const uint4* p0 = reinterpret_cast<const uint4*>(mb + (size_t)kb * sb);
    const uint4* p1 = reinterpret_cast<const uint4*>(mb + (size_t)k1 * sb);
    auto swapped = [](uint32_t x) { return __byte_perm(x, 0u, 0x1032); };
#pragma unroll
    for (int c = 0; c < 32; c += 16) {
      uint4 b0[8], b1[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        b0[i] = __ldg(p0 + c / 2 + i);
        b1[i] = __ldg(p1 + c / 2 + i);
      }
      uint32_t hit = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if ((a0.x & swapped(b0[i].x)) | (a0.y & swapped(b0[i].y)) | (a1.x & swapped(b1[i].x)) |
            (a1.y & swapped(b1[i].y)))
          hit |= 1u << (2 * i);
        if ((a0.x & swapped(b0[i].z)) | (a0.y & swapped(b0[i].w)) | (a1.x & swapped(b1[i].z)) |
            (a1.y & swapped(b1[i].w)))
          hit |= 2u << (2 * i);
      }
      open &= ~(hit << c);
    }
    if (__all_sync(0xffffffffu, open == 0u)) return 0u;
  }
  uint32_t zero = open;  // open ones with no term found so far
  for (int kb = 0; kb < nkb; ++kb) {
    const uint32_t a = has_row ? __ldg(na + (size_t)kb * sa) * 0x10001u : 0u;
    const uint4* p = reinterpret_cast<const uint4*>(nb + (size_t)kb * sb);
    uint32_t hit = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint4 b = __ldg(p + i);
      const uint32_t w[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (a & w[j] & 0xFFFFu) hit |= 1u << (8 * i + 2 * j);
        if (a & w[j] & 0xFFFF0000u) hit |= 2u << (8 * i + 2 * j);
      }
    }
    zero &= ~hit;
    if (__all_sync(0xffffffffu, zero == 0u)) break;
  }
  return open & ~zero;
}

__global__ void __launch_bounds__(NTHREADS, 1)
    gemm_digits_kernel(const DigOperand* __restrict__ ops, const DigSeg* __restrict__ segs,
                       const DigTask* __restrict__ tasks, int ntasks, const unsigned char* __restrict__ pool,
                       const unsigned char* __restrict__ last,
                       const int* __restrict__ exps, const DigMask* __restrict__ masks,
                       const uint16_t* __restrict__ nonzero, int by_entry,
                       int* __restrict__ special, int nops, unsigned char* __restrict__ flag,
                       uint32_t* __restrict__ miss, int* __restrict__ left_blocks, double* __restrict__ scratch,
                       int* __restrict__ err,
                       unsigned long long wait_ns) {
  extern __shared__ unsigned char smraw[];
  __shared__ __align__(8) uint64_t bar[B_COUNT];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, consumed;
  __shared__ Meta meta[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = (smem_u32(smraw) + 1023u) & ~1023u;
  volatile int* abort = &abort_flag;
  auto give_up = [&]() {
    *abort = 1;
    *(volatile int*)err = 1;
  };
  if (tid == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[B_FULL + i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[B_EMPTY + i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[B_SF])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 256;" ::"r"(smem_u32(&bar[B_SE])));
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 32;" ::"r"(smem_u32(&bar[B_MF + i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 256;" ::"r"(smem_u32(&bar[B_ME + i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bar[B_DONE])));
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_flag = 0;
    consumed = 0;
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  int produced = 0;

  if (warp < 4) {
    // registers: 128 (56 + 2 x 224) = 384 x 168, what the block was launched with
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 0) {
      // ---------------------------------------------------------- producer
      // lanes 0..8 copy digit `lane` of the A tile, lanes 9..17 of the B tile
      int q = 0;
      bool ok = true;
      const int s = lane < kDigSlices ? lane : lane - kDigSlices;
      for (int t = blockIdx.x; ok && t < ntasks; t += gridDim.x) {
        const int r0 = tasks[t].r0, c0 = tasks[t].c0, sb = tasks[t].seg_begin, sc = tasks[t].seg_count;
        for (int k = sb; ok && k < sb + sc; ++k) {
          const DigOperand &a = ops[segs[k].a], &b = ops[segs[k].b];
          const int na = min(16, a.groups - (r0 >> 3)), nb = min(8, b.groups - (c0 >> 3));
          const uint32_t bslice = (uint32_t)((nb + 1) & ~1) * kDigUnit;  // 16-column steps
          const int nkb = (a.k + 15) >> 4;
          const bool isb = lane >= kDigSlices, tail = s >= kDigSums;
          const int groups = isb ? b.groups : a.groups;
          const long long unit = isb ? b.unit : a.unit;
          const int g0 = (isb ? c0 : r0) >> 3;
          const unsigned char* src = tail ? last + ((size_t)unit / kDigSums + g0) * kDigUnit
                                          : pool + ((size_t)unit + (size_t)s * groups + g0) * kDigUnit;
          const size_t step = (size_t)(tail ? 1 : kDigSums) * groups * kDigUnit;
          const uint32_t bytes = (uint32_t)(isb ? nb : na) * kDigUnit;
          const uint32_t off = isb ? A_BYTES + s * bslice : s * A_SLICE;
          const uint32_t total = (uint32_t)(na + nb) * kDigSlices * kDigUnit;
          for (int kb = 0; kb < nkb; ++kb, src += step) {
            const int st = q % NSTAGE;
            if (!wait_bar(&bar[B_EMPTY + st], (uint32_t)(((q / NSTAGE) & 1) ^ 1), abort, wait_ns)) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            if (lane == 0) arrive_expect(&bar[B_FULL + st], total);
            __syncwarp();
            if (lane < 2 * kDigSlices) bulk_load(sbase + st * STAGE + off, src, bytes, &bar[B_FULL + st]);
            ++q;
          }
        }
      }
      if (!ok && lane == 0) give_up();
      produced = q;
    } else if (warp == 1 && lane == 0) {
      // ---------------------------------------------------------- MMA issuer
      int q = 0, nd = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < ntasks; t += gridDim.x) {
        const int sb = tasks[t].seg_begin, sc = tasks[t].seg_count;
        const int W = tile_width(tasks[t].n - tasks[t].c0);
        const uint32_t bslice = (uint32_t)(W >> 3) * kDigUnit;
        const int wide = 256 / W;  // digits of B per MMA
        for (int k = sb; ok && k < sb + sc; ++k) {
          const int nkb = (ops[segs[k].a].k + 15) >> 4;
          for (int kb = 0; kb < nkb; ++kb) {
            const bool fresh = kb % CHUNK == 0;
            if (fresh && nd > 0 && !wait_bar(&bar[B_SE], (uint32_t)((nd - 1) & 1), abort, wait_ns)) {
              ok = false;
              break;
            }
            const int st = q % NSTAGE;
            if (!wait_bar(&bar[B_FULL + st], (uint32_t)((q / NSTAGE) & 1), abort, wait_ns)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint32_t sa = sbase + st * STAGE, sB = sa + A_BYTES;
            if (W == kDigTileN) {
#pragma unroll
              for (int i = 0; i < kDigSlices; ++i) {
                const uint64_t da = desc(sa + i * A_SLICE);
#pragma unroll
                for (int j = 0; j < kDigSums - i; j += 4) {
                  const int nj = kDigSums - i - j < 4 ? kDigSums - i - j : 4;
                  mma_bf16(tmem + kDigTileN * (i + j), da, desc(sB + j * B_SLICE), idesc(kDigTileN * nj),
                           (fresh && i == 0) ? 0u : 1u);
                }
                // d = 8, into the accumulator of d = 7
                mma_bf16(tmem + kDigTileN * (kDigSums - 1), da, desc(sB + (kDigSums - i) * B_SLICE),
                         idesc(kDigTileN), 1u);
              }
            } else {
              for (int i = 0; i < kDigSlices; ++i) {
                for (int j = 0; j < kDigSums - i; j += wide)
                  mma_bf16(tmem + (uint32_t)(W * (i + j)), desc(sa + i * A_SLICE), desc(sB + j * bslice),
                           idesc(W * min(wide, kDigSums - i - j)), (fresh && i == 0) ? 0u : 1u);
                mma_bf16(tmem + (uint32_t)(W * (kDigSums - 1)), desc(sa + i * A_SLICE),
                         desc(sB + (kDigSums - i) * bslice), idesc(W), 1u);
              }
            }
            commit(&bar[B_EMPTY + st]);
            ++q;
            if (kb + 1 == nkb || kb % CHUNK == CHUNK - 1) {
              commit(&bar[B_SF]);
              ++nd;
            }
          }
        }
      }
      if (!ok) give_up();
      consumed = q;
      commit(&bar[B_DONE]);
      const unsigned long long t0 = global_ns();
      while (!try_wait(&bar[B_DONE], 0u) && global_ns() - t0 < kDrainNs) __nanosleep(64);
    } else if (warp == 2) {
      // ---------------------------------------------------------- segment data
      int q = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < ntasks; t += gridDim.x) {
        const int sb = tasks[t].seg_begin, sc = tasks[t].seg_count;
        for (int k = sb; k < sb + sc; ++k, ++q) {
          const DigSeg sg = segs[k];
          const DigOperand &a = ops[sg.a], &b = ops[sg.b];
          const int K = a.k;
          const int plain = special[sg.a] | special[sg.b];
          ok = __all_sync(0xffffffffu, wait_bar(&bar[B_ME + (q & 1)], (uint32_t)(((q >> 1) & 1) ^ 1), abort, wait_ns));
          if (!ok) break;
          Meta& m = meta[q & 1];
          const int r0 = tasks[t].r0, c0 = tasks[t].c0, mm = tasks[t].m, nn = tasks[t].n;
          for (int i = lane; i < kDigTileM; i += 32) m.ea[i] = r0 + i < mm ? __ldg(&exps[a.eoff + r0 + i]) - 68 : 0;
          for (int i = lane; i < kDigTileN; i += 32) m.eb[i] = c0 + i < nn ? __ldg(&exps[b.eoff + c0 + i]) : 0;
          if (lane == 0) {
            m.t = tasks[t];
            m.alpha = sg.alpha;
            m.ua = a.unit;
            m.ub = b.unit;
            m.sa = 8 * a.groups;
            m.sb = 8 * b.groups;
            m.k = K;
            m.plain = plain;
          }
          arrive(&bar[B_MF + (q & 1)]);
        }
      }
      if (!ok && lane == 0) give_up();
    }
  } else {
    // ------------------------------------------------------------ epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    constexpr int NC = 32;  // columns of a thread
    const int half = (warp - 4) >> 2;
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    double* const turn = reinterpret_cast<double*>(smraw + (sbase - smem_u32(smraw)) + OFF_TURN +
                                                   (warp - 4) * TURN_BYTES);
    int nd = 0, q = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < ntasks; t += gridDim.x) {
      double acc[32];
      double* out = nullptr;
      long long part = -1;
      int W = 0, ldc = 0, nrow = 0, gc = 0, gr0 = 0, sc = 1;
      bool busy = false;  // the warp has outputs of the block
      bool marked = false;
      for (int k = 0; ok && k < sc; ++k, ++q) {
        ok = __all_sync(0xffffffffu, wait_bar(&bar[B_MF + (q & 1)], (uint32_t)((q >> 1) & 1), abort, wait_ns));
        if (!ok) break;
        const Meta& m = meta[q & 1];
        if (k == 0) {
          W = tile_width(m.t.n - m.t.c0);
          sc = m.t.seg_count;
          part = m.t.part;
          ldc = m.t.ldc;
          // the warp's outputs: rows gr0 + 0..31, column gc (lane)
          gr0 = m.t.r0 + (warp & 3) * 32;
          gc = m.t.c0 + half * NC + lane;
          nrow = gc < m.t.n ? max(0, min(32, m.t.m - gr0)) : 0;
          busy = gr0 < m.t.m && m.t.c0 + half * NC < m.t.n;
          out = m.t.C + (size_t)gr0 * ldc + gc;
          // a tile summed by one task starts from C, loaded while the first
          // products run
#pragma unroll
          for (int r = 0; r < 32; ++r) acc[r] = (part < 0 && r < nrow) ? out[(size_t)r * ldc] : 0.0;
        }
        const int nkb = (m.k + 15) >> 4;
        // outputs left to fma_missing_kernel: bit c of a lane's row
        uint32_t left = 0u;
        if (busy && m.plain) {
          left = 0xFFFFFFFFu;
        } else if (busy && by_entry) {
          const int r = gr0 + lane, c0 = m.t.c0 + half * NC;
          left = outputs_left(r < m.t.m, masks + m.ua + r, nonzero + m.ua + r, m.sa, masks + m.ub + c0,
                              nonzero + m.ub + c0, m.sb, nkb, min(NC, m.t.n - c0));
        }
        const int mark = m.t.mark + 8 * k + warp - 4;
        const bool some = __any_sync(0xffffffffu, left != 0u);
        if (some) miss[(size_t)mark * 32 + lane] = left;
        if (lane == 0) flag[mark] = some;
        marked = marked || some;
        // the combined accumulators of row gr0 + lane: h 2^32 + l, in units of
        // 2^(ea + eb)
        long long h[NC];
        uint32_t l[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          h[c] = 0;
          l[c] = 0u;
        }
        for (int kb = 0; kb < nkb; kb += CHUNK) {
          ok = __all_sync(0xffffffffu, wait_bar(&bar[B_SF], (uint32_t)(nd & 1), abort, wait_ns));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
          for (int c = 0; c < NC; c += 4) {
            if (!busy || half * NC + c >= W) break;
            uint32_t v[kDigSums][4];
#pragma unroll
            for (int d = 0; d < kDigSums; ++d) tmem_ld4(lanes + (uint32_t)(W * d + half * NC + c), v[d]);
            asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              // in units of their weights, 2^-8d
              auto S = [&](int d) {
                return __float2int_rn(__uint_as_float(v[d][i]) * __uint_as_float((uint32_t)(127 + 8 * d) << 23));
              };
              long long lo = (long long)l[c + i] + S(7);
              lo = mad_wide(S(6), 1 << 8, lo);
              lo = mad_wide(S(5), 1 << 16, lo);
              lo = mad_wide(S(4), 1 << 24, lo);
              l[c + i] = (uint32_t)lo;
              long long hi = h[c + i] + (int)(lo >> 32);
              hi += S(3);
              hi = mad_wide(S(2), 1 << 8, hi);
              hi = mad_wide(S(1), 1 << 16, hi);
              h[c + i] = mad_wide(S(0), 1 << 24, hi);
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;");
          arrive(&bar[B_SE]);
          ++nd;
        }
        if (!ok) break;
        if (!busy || m.plain) {
          // nothing of the block in this warp's rows and columns: the float64
          // pipe belongs to the others (the 442 launches of a D = 256 sweep, whose
          // blocks are mostly below 128 x 64: 14.7 -> 11.8 ms)
          arrive(&bar[B_ME + (q & 1)]);
          continue;
        }
        double sum[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) sum[c] = c < 16 || half * NC + 16 < W ? combined(h[c], l[c]) : 0.0;
        // bit r: this lane's column of row r is an output of the digits
        uint32_t live = nrow > 0 ? 0xFFFFFFFFu >> (32 - nrow) : 0u;
        if (some) {
#pragma unroll 4
          for (int c = 0; c < 32; ++c) {
            const uint32_t rows = __ballot_sync(0xffffffffu, left >> c & 1u);
            if (lane == c) live &= ~rows;
          }
        }
        const double alpha = m.alpha;
        const int m_rows = m.t.m;
        const int eb = m.eb[half * NC + lane];
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          // rows 16 p ... of the block
          if (lane >> 4 == p) {
#pragma unroll
            for (int c = 0; c < NC; ++c) turn[(lane & 15) * TURN_LD + c] = sum[c];
          }
          __syncwarp();
#pragma unroll
          for (int r = 16 * p; r < 16 * p + 16; ++r) {
            if (r % 8 == 0 && gr0 + r >= m_rows) break;
            // times 2^e: the value is zero or in [1, 2^84), |e| <= 872
            const int e = eb + m.ea[(warp & 3) * 32 + r];
            const double d = turn[(r & 15) * TURN_LD + lane];
            const int hi = __double2hiint(d);
            if (live >> r & 1u)
              acc[r] = fma(alpha, __hiloint2double(hi ? hi + (e << 20) : 0, __double2loint(d)), acc[r]);
          }
          __syncwarp();
        }
        arrive(&bar[B_ME + (q & 1)]);
      }
      if (!ok) break;
      if (marked && lane == 0) left_blocks[atomicAdd(&special[nops], 1)] = 8 * t + warp - 4;
      if (part >= 0) {
        // row-major partial tile of 128 x 64
        double* p = scratch + part + (size_t)((warp & 3) * 32) * kDigTileN + half * NC + lane;
#pragma unroll
        for (int r = 0; r < 32; ++r) p[(size_t)r * kDigTileN] = acc[r];
      } else {
#pragma unroll
        for (int r = 0; r < 32; ++r)
          if (r < nrow) out[(size_t)r * ldc] = acc[r];
      }
    }
    if (!ok && lane == 0) give_up();
  }
  __syncthreads();
  if (warp == 0 && lane == 0 && *abort) {
    // copies still in flight land before the CTA exits
    for (int q = consumed; q < produced; ++q) {
      const unsigned long long t0 = global_ns();
      while (!try_wait(&bar[B_FULL + q % NSTAGE], (uint32_t)((q / NSTAGE) & 1)) && global_ns() - t0 < kDrainNs)
        __nanosleep(64);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// What gemm_digits_kernel left out, added to the tiles by float64 FMAs.  A CTA
// takes 16 x 32 outputs of a block with marks and its marked segments in order; the missing
// outputs are dealt to the threads one by one, two each, or a few threads each
// (along k) where there are few.  Bound by the float64 pipe (two FMAs a clock
// and SM) where whole blocks are missing: two shared-memory reads an FMA, one
// along the lanes and one broadcast, are a fifth of its time.  Where single
// outputs are missing, by the latency of the loads, so two steps of 64 columns
// are in flight; and blocks this small, taken from a list, spread what is missing
// in a corner of a matrix over the SMs (exchange of 200 orbitals: 970 us with
// blocks dealt by their place, 435 from the list).  Measured, whole calls with
// every operand graded: 400 x 400 x 400 0.34 ms, 601 of 200 x 200 x 200 14.3 ms
// (0.95 and 18.4 ms by gemm_f64_kernel alone).  Without marks 1.3 us.
constexpr int FIX_THREADS = 256, FIX_ROWS = 16, FIX_COLS = 32, FIX_K = 64, FIX_LD = FIX_K + 1;
constexpr int FIX_CTAS = 4;
constexpr int FIX_OUT = FIX_ROWS * FIX_COLS / FIX_THREADS;
constexpr int FIX_STAGE = (FIX_ROWS + FIX_COLS) * FIX_LD, FIX_SMEM = 2 * FIX_STAGE * (int)sizeof(double);

__device__ __forceinline__ void copy8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// rows [r0, r0 + nr) and columns [k0, k0 + kn) of an operand, row r at r FIX_LD
template <int ROWS>
__device__ __forceinline__ void fix_stage(double* dst, const DigOperand& o, int r0, int nr, int k0, int kn) {
  for (int e = threadIdx.x; e < ROWS * FIX_K; e += FIX_THREADS) {
    const int r = o.trans ? e % ROWS : e / FIX_K, k = o.trans ? e / ROWS : e % FIX_K;
    if (r < nr && k < kn)
      copy8(dst + r * FIX_LD + k,
            o.src + (o.trans ? (size_t)(k0 + k) * o.ld + r0 + r : (size_t)(r0 + r) * o.ld + k0 + k));
  }
}

__global__ void __launch_bounds__(FIX_THREADS, FIX_CTAS)
    fma_missing_kernel(const DigOperand* __restrict__ ops, const DigSeg* __restrict__ segs,
                       const DigTask* __restrict__ tasks, const int* __restrict__ nleft,
                       const int* __restrict__ left, const unsigned char* __restrict__ flag,
                       const uint32_t* __restrict__ miss, double* __restrict__ scratch) {
  // 16 rows a CTA, or 8 or 4 where that makes fewer than two units a CTA: 16 x 32
  // outputs of a 150 x 150 product are 20 us of an SM's float64 pipe (33 -> 14 us;
  // exchange of 200 orbitals 590 -> 435 us against one unit a CTA)
  const int blocks = *nleft;
  int rows = FIX_ROWS;
  while (rows > 4 && blocks * (32 / rows) < 2 * (int)gridDim.x) rows /= 2;
  const int per = 32 / rows, units = blocks * per;
  extern __shared__ double fix[];
  __shared__ unsigned short list[FIX_ROWS * FIX_COLS];
  __shared__ int count;
  const int tid = threadIdx.x;
  for (int u = blockIdx.x; u < units; u += gridDim.x) {
    const int block = left[u / per], w = block & 7, sub = u % per * rows;  // the mark, first row of it
    const DigTask t = tasks[block >> 3];
    const int r0 = t.r0 + (w & 3) * 32 + sub, c0 = t.c0 + (w >> 2) * FIX_COLS;
    const int nr = min(rows, t.m - r0), nc = min(FIX_COLS, t.n - c0);
    if (nr <= 0) continue;
    for (int s = 0; s < t.seg_count; ++s) {
      const int mark = t.mark + 8 * s + w;
      if (!flag[mark]) continue;
      const DigSeg sg = segs[t.seg_begin + s];
      const DigOperand a = ops[sg.a], b = ops[sg.b];
      __syncthreads();  // the list and the stages are free, the outputs of the segment before visible
      if (tid < 32) {
        uint32_t bits = tid < nr ? miss[(size_t)mark * 32 + sub + tid] & (0xFFFFFFFFu >> (32 - nc)) : 0u;
        int at = __popc(bits);
#pragma unroll
        for (int d = 1; d < 32; d *= 2) {
          const int x = __shfl_up_sync(0xffffffffu, at, d);
          if (tid >= d) at += x;
        }
        if (tid == 31) count = at;
        at -= __popc(bits);
        for (; bits; bits &= bits - 1) list[at++] = (unsigned short)(tid * FIX_COLS + __ffs(bits) - 1);
      }
      __syncthreads();
      const int n = count;
      if (n == 0) continue;
      // lanes of an output: a power of two, at most eight
      int lanes = 1;
      while (lanes < 8 && 2 * lanes * n <= FIX_THREADS) lanes *= 2;
      const int step = FIX_THREADS / lanes, first = tid / lanes, sub_k = tid - first * lanes;
      double acc[FIX_OUT];
      int ao[FIX_OUT], bo[FIX_OUT];
#pragma unroll
      for (int q = 0; q < FIX_OUT; ++q) {
        const int i = first + q * step, e = i < n ? list[i] : 0;
        acc[q] = 0.0;
        ao[q] = e / FIX_COLS * FIX_LD;
        bo[q] = FIX_ROWS * FIX_LD + e % FIX_COLS * FIX_LD;
      }
      const int nq = first >= n ? 0 : min(FIX_OUT, (n - first + step - 1) / step);
      auto stage = [&](int k0) {
        double* const dst = fix + (k0 / FIX_K & 1) * FIX_STAGE;
        if (k0 < a.k) {
          fix_stage<FIX_ROWS>(dst, a, r0, nr, k0, min(FIX_K, a.k - k0));
          fix_stage<FIX_COLS>(dst + FIX_ROWS * FIX_LD, b, c0, nc, k0, min(FIX_K, a.k - k0));
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
      stage(0);
      for (int k0 = 0; k0 < a.k; k0 += FIX_K) {
        const int kn = min(FIX_K, a.k - k0);
        const double* x = fix + (k0 / FIX_K & 1) * FIX_STAGE;
        stage(k0 + FIX_K);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (lanes == 1 && nq == FIX_OUT) {
#pragma unroll 4
          for (int k = 0; k < kn; ++k)
#pragma unroll
            for (int q = 0; q < FIX_OUT; ++q) acc[q] = fma(x[ao[q] + k], x[bo[q] + k], acc[q]);
        } else if (nq > 0) {
#pragma unroll 4
          for (int k = sub_k; k < kn; k += lanes) acc[0] = fma(x[ao[0] + k], x[bo[0] + k], acc[0]);
        }
        __syncthreads();
      }
      if (lanes > 1)
        for (int d = 1; d < lanes; d *= 2) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], d);
#pragma unroll
      for (int q = 0; q < FIX_OUT; ++q) {
        if (q >= nq || sub_k != 0) break;
        const int e = list[first + q * step], r = e / FIX_COLS, c = e % FIX_COLS;
        double* const out = t.part >= 0
                                ? scratch + t.part + (size_t)(r0 - t.r0 + r) * kDigTileN + (c0 - t.c0) + c
                                : t.C + (size_t)(r0 + r) * t.ldc + c0 + c;
        *out = fma(sg.alpha, acc[q], *out);
      }
    }
  }
}

// C += the partial tiles of one output tile, in order; a CTA sums 4 rows
__global__ void __launch_bounds__(256) reduce_digits_kernel(const DigReduce* __restrict__ reds,
                                                            const double* __restrict__ scratch) {
  const DigReduce rd = reds[blockIdx.x];
  const int c = threadIdx.x & (kDigTileN - 1), gc = rd.c0 + c;
  const int r = blockIdx.y * 4 + (int)(threadIdx.x >> 6), gr = rd.r0 + r;
  if (gr >= rd.m || gc >= rd.n) return;
  const double* p = scratch + rd.part0 + (size_t)r * kDigTileN + c;
  double s = 0.0;
#pragma unroll 4
  for (int i = 0; i < rd.nparts; ++i) s += p[(size_t)i * kDigTileM * kDigTileN];
  rd.C[(size_t)gr * rd.ldc + gc] += s;
}

}  // namespace

void dig_launch(const DigLaunch& L, cudaStream_t st) {
  cudaError_t e = ensure_smem_attr((const void*)gemm_digits_kernel, SMEM_BYTES);
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit gemm attribute: ") + cudaGetErrorString(e));
  e = ensure_smem_attr((const void*)fma_missing_kernel, FIX_SMEM);
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit remainder attribute: ") + cudaGetErrorString(e));
  split_digits_kernel<<<L.nsplits, SPLIT_THREADS, 0, st>>>(L.ops, L.splits, L.pool, L.last, L.exps, L.masks, L.nonzero,
                                                               L.special);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit split: ") + cudaGetErrorString(e));
  gemm_digits_kernel<<<std::min(L.sms, L.ntasks), NTHREADS, SMEM_BYTES, st>>>(
      L.ops, L.segs, L.tasks, L.ntasks, L.pool, L.last, L.exps, L.masks, L.nonzero, L.by_entry, L.special, L.nops, L.flag, L.miss,
      L.left, L.scratch, L.err, L.wait_ns);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit gemm: ") + cudaGetErrorString(e));
  fma_missing_kernel<<<std::min(L.sms * FIX_CTAS, L.ntasks * 64), FIX_THREADS, FIX_SMEM, st>>>(
      L.ops, L.segs, L.tasks, L.special + L.nops, L.left, L.flag, L.miss, L.scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit remainder: ") + cudaGetErrorString(e));
  if (L.nreds > 0) {
    reduce_digits_kernel<<<dim3(L.nreds, kDigTileM / 4), 256, 0, st>>>(L.reds, L.scratch);
    e = cudaGetLastError();
    if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit reduce: ") + cudaGetErrorString(e));
  }
}

}  // namespace dmrg
