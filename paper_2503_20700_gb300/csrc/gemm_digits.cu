// Float64 grouped GEMM by exact digit products on tcgen05 (gemm_digits.cuh).
//
// gemm_digits_kernel is persistent (one CTA per SM, tasks dealt longest
// first).  A k-step of 16 brings the eight digits of 128 rows of op(A) and 64
// columns of op(B) (48 KB, 16 bulk copies) into one of three stages; digit i
// of A meets the digits 0..7-i of B, stacked along N, so one MMA of N = 256
// covers four digits of B and its output columns are the accumulators
// i..i+3: 12 MMAs and 1152 tensor clocks a k-step.  The eight accumulators
// (128 x 64 FP32 each) fill TMEM.
//
// What bounds it: shared memory for long segments (a k-step's 12 MMAs read
// 120 KB and its copies write 48 KB: 1500 clocks, 1152 on the tensor pipe
// alone), the float64 pipe for short ones (three operations per output and
// segment at two a clock and SM, 12300 clocks a tile).  The tile is 128 x 64
// because eight accumulators of that size are all of TMEM; N = 64 alone would
// read shared memory at 48 clocks per 32-clock MMA, which the stacked form
// avoids.  Measured, 601 products of 200 x 200 x 200 (the rotation of 600
// Cholesky vectors): 0.43 ms and 0.17 ms for the split, 16 TFLOP/s of float64;
// the FMA kernel needs 13 ms (0.74 TFLOP/s, 1.25 nominal peak).
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
// per epilogue warp: 32 x 32 outputs, turned from row-per-lane (TMEM) to
// column-per-lane (coalesced C)
constexpr int TURN_LD = 33;
constexpr int OFF_TURN = NSTAGE * STAGE, TURN_BYTES = 32 * TURN_LD * 8;
constexpr int SMEM_BYTES = OFF_TURN + 8 * TURN_BYTES + 1024;
constexpr int CHUNK = 16;  // k-steps of 16 between drains: 256 exact terms
constexpr int NTHREADS = 384;
constexpr unsigned long long kDrainNs = 2000000000ull;  // what a CTA that gave up waits for its own work in flight
constexpr int kExpRange = 400;
constexpr int kGraded = 8;  // the largest product may lie 2^8 below the product of the maxima

enum { B_FULL = 0, B_EMPTY = B_FULL + NSTAGE, B_SF = B_EMPTY + NSTAGE, B_SE, B_MF, B_ME = B_MF + 2,
       B_DONE = B_ME + 2, B_COUNT };

// what the epilogue needs of a segment, gathered one segment ahead by a warp
// of its own (the dependent loads task - segment - operand - column maxima
// took a third of the epilogue's time)
struct Meta {
  DigTask t;
  double alpha;
  int a, b, k, plain;
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
// the eight bytes of u (digit + 128 each, digit 0 on top) as bf16 pairs: word
// s of `w` gets digit s of this element in its half `half`
__device__ __forceinline__ float digit_float(uint32_t word, int byte) {
  // 2^23 + byte, minus 2^23 + 128
  return __uint_as_float(__byte_perm(word, 0x4B000000u, 0x7440 + byte)) - 8388736.0f;
}

// 32 rows of one operand per CTA: row maxima, then the digits.  Bound by the
// latency of its loads for the matrices of a sweep and by HBM and the integer
// pipe together for large ones (8 B read twice, 16 B written, about 35
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
                                                                     int* __restrict__ exps,
                                                                     uint2* __restrict__ kmax,
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
  unsigned char* const base = pool + (size_t)o.unit * kDigUnit + (size_t)g * kDigUnit + kc * 128 + (lane & 7) * 16;
  for (int kb = warp >> 1; kb < nkb; kb += KSTEP) {
    const int c0 = kb * 16 + kc * 8;
    double x[8];
    load8(o, r, c0, x);
    uint32_t w[kDigSlices][4];
    unsigned rel = 0u, top = 0u;  // column c0 + (lane & 7), once the loop is done
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      float f[2][kDigSlices];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(x[i + q]);
        const int be = (int)((bits >> 52) & 0x7FF);
        unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | 1ull << 52;
        const int sh = be - be_row + 9;  // at most 9
        if (be == 0 || sh < -54) m = 0;
        else if (sh >= 0) m <<= sh;
        else m = (m + (1ull << (-sh - 1))) >> -sh;
        const unsigned long long F = (long long)bits < 0 ? 0ull - m : m;
        const unsigned long long u = F + 0x8080808080808080ull;
        const uint32_t uh = (uint32_t)(u >> 32), ul = (uint32_t)u;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          f[q][s] = digit_float(uh, 3 - s);
          f[q][4 + s] = digit_float(ul, 3 - s);
        }
        // largest entry of the column over the eight rows: relative to its
        // row's maximum (shifted by 4096, so that 0 is a zero) and absolute
        unsigned a = be ? (unsigned)(4096 + be - be_row) : 0u, b = (unsigned)be;
#pragma unroll
        for (int d = 1; d < 8; d *= 2) {
          a = max(a, __shfl_xor_sync(0xffffffffu, a, d));
          b = max(b, __shfl_xor_sync(0xffffffffu, b, d));
        }
        if ((lane & 7) == i + q) {
          rel = a;
          top = b;
        }
      }
#pragma unroll
      for (int s = 0; s < kDigSlices; ++s)
        w[s][i >> 1] = __byte_perm(__float_as_uint(f[0][s]), __float_as_uint(f[1][s]), 0x7632);
    }
    if (stored) {
#pragma unroll
      for (int s = 0; s < kDigSlices; ++s)
        *reinterpret_cast<uint4*>(base + ((size_t)kb * kDigSlices + s) * o.groups * kDigUnit) =
            make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
    }
    // the two row groups of the warp, then all rows of the operand
    rel = max(rel, __shfl_xor_sync(0xffffffffu, rel, 16));
    top = max(top, __shfl_xor_sync(0xffffffffu, top, 16));
    const int c = c0 + (lane & 7);
    if (lane < 16 && c < o.k && rel) {
      atomicMax(&kmax[o.koff + c].x, rel);
      atomicMax(&kmax[o.koff + c].y, top);
    }
  }
}

// ---------------------------------------------------------------- products
__global__ void __launch_bounds__(NTHREADS, 1)
    gemm_digits_kernel(const DigOperand* __restrict__ ops, const DigSeg* __restrict__ segs,
                       const DigTask* __restrict__ tasks, int ntasks, const unsigned char* __restrict__ pool,
                       const int* __restrict__ exps, const uint2* __restrict__ kmax,
                       int* __restrict__ special, int nops, unsigned char* __restrict__ flag,
                       uint32_t* __restrict__ miss, double* __restrict__ scratch, int* __restrict__ err,
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
      // lanes 0..7 copy digit `lane` of the A tile, lanes 8..15 of the B tile
      int q = 0;
      bool ok = true;
      const int s = lane & 7;
      for (int t = blockIdx.x; ok && t < ntasks; t += gridDim.x) {
        const int r0 = tasks[t].r0, c0 = tasks[t].c0, sb = tasks[t].seg_begin, sc = tasks[t].seg_count;
        for (int k = sb; ok && k < sb + sc; ++k) {
          const DigOperand &a = ops[segs[k].a], &b = ops[segs[k].b];
          const int na = min(16, a.groups - (r0 >> 3)), nb = min(8, b.groups - (c0 >> 3));
          const uint32_t bslice = (uint32_t)((nb + 1) & ~1) * kDigUnit;  // 16-column steps
          const int nkb = (a.k + 15) >> 4;
          const bool isb = lane >= 8;
          const int groups = isb ? b.groups : a.groups;
          const unsigned char* src =
              pool + ((isb ? b.unit : a.unit) + (size_t)s * groups + ((isb ? c0 : r0) >> 3)) * kDigUnit;
          const size_t step = (size_t)kDigSlices * groups * kDigUnit;
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
            if (lane < 16) bulk_load(sbase + st * STAGE + off, src, bytes, &bar[B_FULL + st]);
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
                for (int j = 0; j < kDigSlices - i; j += 4) {
                  const int nj = kDigSlices - i - j < 4 ? kDigSlices - i - j : 4;
                  mma_bf16(tmem + kDigTileN * (i + j), da, desc(sB + j * B_SLICE), idesc(kDigTileN * nj),
                           (fresh && i == 0) ? 0u : 1u);
                }
              }
            } else {
              for (int i = 0; i < kDigSlices; ++i)
                for (int j = 0; j < kDigSlices - i; j += wide)
                  mma_bf16(tmem + (uint32_t)(W * (i + j)), desc(sa + i * A_SLICE), desc(sB + j * bslice),
                           idesc(W * min(wide, kDigSlices - i - j)), (fresh && i == 0) ? 0u : 1u);
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
          // may the digits be used: the largest products of the segment against
          // the products of the maxima (no overlapping column: an exact zero)
          unsigned rel = 0u, top = 0u, amax = 0u, bmax = 0u;
          const uint2 *ka = kmax + a.koff, *kb = kmax + b.koff;
#pragma unroll 4
          for (int c = lane; c < K; c += 32) {
            const uint2 x = __ldg(ka + c), y = __ldg(kb + c);
            if (x.x && y.x) {
              rel = max(rel, x.x + y.x);
              top = max(top, x.y + y.y);
            }
            amax = max(amax, x.y);
            bmax = max(bmax, y.y);
          }
          rel = __reduce_max_sync(0xffffffffu, rel);
          top = __reduce_max_sync(0xffffffffu, top);
          amax = __reduce_max_sync(0xffffffffu, amax);
          bmax = __reduce_max_sync(0xffffffffu, bmax);
          const int plain = (special[sg.a] | special[sg.b]) ||
                            (rel && (rel + kGraded < 8192u || top + kGraded < amax + bmax));
          ok = __all_sync(0xffffffffu, wait_bar(&bar[B_ME + (q & 1)], (uint32_t)(((q >> 1) & 1) ^ 1), abort, wait_ns));
          if (!ok) break;
          Meta& m = meta[q & 1];
          const int r0 = tasks[t].r0, c0 = tasks[t].c0, mm = tasks[t].m, nn = tasks[t].n;
          for (int i = lane; i < kDigTileM; i += 32) m.ea[i] = r0 + i < mm ? __ldg(&exps[a.eoff + r0 + i]) - 68 : 0;
          for (int i = lane; i < kDigTileN; i += 32) m.eb[i] = c0 + i < nn ? __ldg(&exps[b.eoff + c0 + i]) : 0;
          if (lane == 0) {
            m.t = tasks[t];
            m.alpha = sg.alpha;
            m.a = sg.a;
            m.b = sg.b;
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
            uint32_t v[kDigSlices][4];
#pragma unroll
            for (int d = 0; d < kDigSlices; ++d) tmem_ld4(lanes + (uint32_t)(W * d + half * NC + c), v[d]);
            asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              auto S = [&](int d) { return __float2int_rn(__uint_as_float(v[d][i])); };
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
        const int mark = m.t.mark + 8 * k + warp - 4;
        const bool left = busy && m.plain;  // to fma_missing_kernel
        if (lane == 0) {
          flag[mark] = left;
          if (left) special[nops] = 1;
        }
        if (left) {
          miss[(size_t)mark * 32 + lane] = 0xFFFFFFFFu;
          arrive(&bar[B_ME + (q & 1)]);
          continue;
        }
        if (!busy) {
          // nothing of the block in this warp's rows and columns: the float64
          // pipe belongs to the others (the 442 launches of a D = 256 sweep, whose
          // blocks are mostly below 128 x 64: 14.7 -> 11.8 ms)
          arrive(&bar[B_ME + (q & 1)]);
          continue;
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          if (c % 16 == 0 && half * NC + c >= W) break;
          turn[lane * TURN_LD + c] = combined(h[c], l[c]);
        }
        __syncwarp();
        const double alpha = m.alpha;
        const int m_rows = m.t.m;
        const int eb = m.eb[half * NC + lane];
#pragma unroll
        for (int r = 0; r < 32; ++r) {
          if (r % 8 == 0 && gr0 + r >= m_rows) break;
          // times 2^e: the value is zero or in [1, 2^84), |e| <= 872
          const int e = eb + m.ea[(warp & 3) * 32 + r];
          const double d = turn[r * TURN_LD + lane];
          const int hi = __double2hiint(d);
          if (r < nrow) acc[r] = fma(alpha, __hiloint2double(hi ? hi + (e << 20) : 0, __double2loint(d)), acc[r]);
        }
        __syncwarp();
        arrive(&bar[B_ME + (q & 1)]);
      }
      if (!ok) break;
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

// What gemm_digits_kernel left out: per mark, the missing outputs of a 32 x 32
// block are dealt to the threads one by one, four each, and their products
// added to the tile by float64 FMAs.  Bound by the float64 pipe (two FMAs a
// clock and SM) where whole blocks are missing: two shared-memory reads an FMA,
// one along the lanes and one broadcast, are a fifth of its time, and blocks of
// 32 x 32 spread even a single product over the SMs.  Measured, whole calls with
// every operand graded: 400 x 400 x 400 2.19 -> 0.42 ms, 601 of 200 x 200 x 200
// 39.6 -> 19.2 ms (one in ten graded: 9.5 -> 7.0) against FMAs on unstaged
// operands in the epilogue of the digit kernel; gemm_f64_kernel alone takes 0.96
// and 18.4 ms.  Without marks the launch costs 1.3 us and 2 us of the host.
constexpr int FIX_THREADS = 256, FIX_K = 64, FIX_LD = FIX_K + 1, FIX_OUT = 1024 / FIX_THREADS, FIX_CTAS = 5;
__global__ void __launch_bounds__(FIX_THREADS, FIX_CTAS)
    fma_missing_kernel(const DigOperand* __restrict__ ops, const DigSeg* __restrict__ segs,
                       const DigTask* __restrict__ tasks, int ntasks, const int* __restrict__ any,
                       const unsigned char* __restrict__ flag, const uint32_t* __restrict__ miss,
                       double* __restrict__ scratch) {
  if (*any == 0) return;
  __shared__ double As[32 * FIX_LD], Bs[32 * FIX_LD];
  __shared__ unsigned short list[1024];
  __shared__ int count;
  const int tid = threadIdx.x;
  for (int u = blockIdx.x; u < ntasks * 8; u += gridDim.x) {
    const int w = u / ntasks;  // every CTA meets all eight: the last ones of a ragged tile are empty
    const DigTask t = tasks[u - w * ntasks];
    const int r0 = t.r0 + (w & 3) * 32, c0 = t.c0 + (w >> 2) * 32;
    const int nr = min(32, t.m - r0), nc = min(32, t.n - c0);
    if (nr <= 0 || nc <= 0) continue;
    for (int s = 0; s < t.seg_count; ++s) {
      const int mark = t.mark + 8 * s + w;
      if (!flag[mark]) continue;
      __syncthreads();  // the list and the tiles are free, the block's outputs visible
      if (tid < 32) {
        uint32_t bits = tid < nr ? miss[(size_t)mark * 32 + tid] & (0xFFFFFFFFu >> (32 - nc)) : 0u;
        int at = __popc(bits);
#pragma unroll
        for (int d = 1; d < 32; d *= 2) {
          const int x = __shfl_up_sync(0xffffffffu, at, d);
          if (tid >= d) at += x;
        }
        if (tid == 31) count = at;
        at -= __popc(bits);
        for (; bits; bits &= bits - 1) list[at++] = (unsigned short)(tid * 32 + __ffs(bits) - 1);
      }
      __syncthreads();
      const int n = count;
      const DigSeg sg = segs[t.seg_begin + s];
      const DigOperand a = ops[sg.a], b = ops[sg.b];
      double acc[FIX_OUT];
      int ao[FIX_OUT], bo[FIX_OUT];
#pragma unroll
      for (int q = 0; q < FIX_OUT; ++q) {
        const int i = tid + q * FIX_THREADS, e = i < n ? list[i] : 0;
        acc[q] = 0.0;
        ao[q] = (e >> 5) * FIX_LD;
        bo[q] = (e & 31) * FIX_LD;
      }
      const int nq = (n - tid + FIX_THREADS - 1) / FIX_THREADS;  // of this thread
      for (int k0 = 0; k0 < a.k; k0 += FIX_K) {
        const int kn = min(FIX_K, a.k - k0);
        for (int e = tid; e < 32 * FIX_K; e += FIX_THREADS) {
          const int r = a.trans ? e & 31 : e / FIX_K, k = a.trans ? e >> 5 : e % FIX_K;
          if (r < nr && k < kn) As[r * FIX_LD + k] = sg.alpha * elem(a, r0 + r, k0 + k);
        }
        for (int e = tid; e < 32 * FIX_K; e += FIX_THREADS) {
          const int c = b.trans ? e & 31 : e / FIX_K, k = b.trans ? e >> 5 : e % FIX_K;
          if (c < nc && k < kn) Bs[c * FIX_LD + k] = elem(b, c0 + c, k0 + k);
        }
        __syncthreads();
        if (nq == FIX_OUT) {
#pragma unroll 4
          for (int k = 0; k < kn; ++k)
#pragma unroll
            for (int q = 0; q < FIX_OUT; ++q) acc[q] = fma(As[ao[q] + k], Bs[bo[q] + k], acc[q]);
        } else {
#pragma unroll
          for (int q = 0; q < FIX_OUT - 1; ++q)
            if (q < nq)
              for (int k = 0; k < kn; ++k) acc[q] = fma(As[ao[q] + k], Bs[bo[q] + k], acc[q]);
        }
        __syncthreads();
      }
#pragma unroll
      for (int q = 0; q < FIX_OUT; ++q) {
        if (q >= nq) break;
        const int e = list[tid + q * FIX_THREADS], r = e >> 5, c = e & 31;
        double* const out = t.part >= 0
                                ? scratch + t.part + (size_t)(r0 - t.r0 + r) * kDigTileN + (c0 - t.c0) + c
                                : t.C + (size_t)(r0 + r) * t.ldc + c0 + c;
        *out += acc[q];
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
  split_digits_kernel<<<L.nsplits, SPLIT_THREADS, 0, st>>>(L.ops, L.splits, L.pool, L.exps, L.kmax, L.special);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit split: ") + cudaGetErrorString(e));
  gemm_digits_kernel<<<std::min(L.sms, L.ntasks), NTHREADS, SMEM_BYTES, st>>>(
      L.ops, L.segs, L.tasks, L.ntasks, L.pool, L.exps, L.kmax, L.special, L.nops, L.flag, L.miss, L.scratch, L.err,
      L.wait_ns);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit gemm: ") + cudaGetErrorString(e));
  fma_missing_kernel<<<std::min(L.sms * FIX_CTAS, L.ntasks * 8), FIX_THREADS, 0, st>>>(
      L.ops, L.segs, L.tasks, L.ntasks, L.special + L.nops, L.flag, L.miss, L.scratch);
  e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit remainder: ") + cudaGetErrorString(e));
  if (L.nreds > 0) {
    reduce_digits_kernel<<<dim3(L.nreds, kDigTileM / 4), 256, 0, st>>>(L.reds, L.scratch);
    e = cudaGetLastError();
    if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: digit reduce: ") + cudaGetErrorString(e));
  }
}

}  // namespace dmrg
