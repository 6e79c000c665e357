// Fused H_eff psi kernels (see hpsi_fused.cuh).
#include <algorithm>
#include <stdexcept>
#include <string>

#include "hpsi_fused.cuh"
#include "hpsi_noalloc.hpp"
#include "kattr.hpp"
#include "tf32_bits.cuh"

namespace dmrg {

namespace {

constexpr int T = 64;   // tile edge of sigma and of the psi column chunk
constexpr int KS = 16;  // k-step of the staged operand tiles

// ---------------------------------------------------------------- helpers
__device__ __forceinline__ uint32_t tf32(float x) { return tf32_round(x); }
// by integers: the float64 pipe converts two numbers a clock and SM, which bound
// this kernel (a call with sectors of some tens, 1258 -> 831 us)
__device__ __forceinline__ void split64(double x, uint32_t& hi, uint32_t& lo) {
  float h, l;
  split_tf32(x, h, l);
  hi = __float_as_uint(h);
  lo = __float_as_uint(l);
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// element (r, c) of op(A) (m x k); op = identity when trans == 0
__device__ __forceinline__ double ldA(const HpsiItem& it, int r, int c) {
  return it.transA ? it.A[(size_t)c * it.lda + r] : it.A[(size_t)r * it.lda + c];
}
// element (n, k) of the right operand as used in X B^T
__device__ __forceinline__ double ldB(const HpsiItem& it, int n, int k) {
  return it.transB ? it.B[(size_t)k * it.ldb + n] : it.B[(size_t)n * it.ldb + k];
}

// shared-memory layout (32-bit words) of the TF32 kernel
constexpr int LDS = KS + 4;      // padded row of a 16-wide staged tile
constexpr int LDX = T + 4;       // padded row of the X tile
constexpr int SM_AH = 0;
constexpr int SM_AL = SM_AH + T * LDS;
constexpr int SM_PH = SM_AL + T * LDS;  // P stored n-major: [n][k]
constexpr int SM_PL = SM_PH + T * LDS;
constexpr int SM_BH = SM_PL + T * LDS;  // B stored n-major: [n][k]
constexpr int SM_BL = SM_BH + T * LDS;
constexpr int SM_XH = SM_BL + T * LDS;  // X stored m-major: [m][k]
constexpr int SM_XL = SM_XH + T * LDX;
constexpr int SM_WORDS = SM_XL + T * LDX;

// warp tile: 16 rows x 32 cols of the 64 x 64 tile; acc[nt][q] per mma.sync fragment
__device__ __forceinline__ void warp_mma_k16(float (&acc)[4][4], const uint32_t* Ah, const uint32_t* Al,
                                             int lda_s, const uint32_t* Bh, const uint32_t* Bl, int ldb_s,
                                             int kofs, int wm, int wn, int gid, int tig) {
#pragma unroll
  for (int ks = 0; ks < KS; ks += 8) {
    const int r = wm * 16 + gid;
    const int k = kofs + ks + tig;
    uint32_t ah[4] = {Ah[r * lda_s + k], Ah[(r + 8) * lda_s + k], Ah[r * lda_s + k + 4], Ah[(r + 8) * lda_s + k + 4]};
    uint32_t al[4] = {Al[r * lda_s + k], Al[(r + 8) * lda_s + k], Al[r * lda_s + k + 4], Al[(r + 8) * lda_s + k + 4]};
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) {
      const int c = wn * 32 + nt * 8 + gid;
      const int kb = ks + tig;
      uint32_t bh[2] = {Bh[c * ldb_s + kb], Bh[c * ldb_s + kb + 4]};
      uint32_t bl[2] = {Bl[c * ldb_s + kb], Bl[c * ldb_s + kb + 4]};
      mma(acc[nt], al, bh);
      mma(acc[nt], ah, bl);
      mma(acc[nt], ah, bh);
    }
  }
}

__global__ void __launch_bounds__(256) hpsi_tf32x3_kernel(const HpsiBlock* __restrict__ blocks,
                                                          const HpsiItem* __restrict__ items,
                                                          const HpsiTask* __restrict__ tasks,
                                                          double* __restrict__ scratch) {
  extern __shared__ uint32_t sm[];
  uint32_t* Ah = sm + SM_AH;
  uint32_t* Al = sm + SM_AL;
  uint32_t* Ph = sm + SM_PH;
  uint32_t* Pl = sm + SM_PL;
  uint32_t* Bh = sm + SM_BH;
  uint32_t* Bl = sm + SM_BL;
  uint32_t* Xh = sm + SM_XH;
  uint32_t* Xl = sm + SM_XL;
  const HpsiTask tk = tasks[blockIdx.x];
  const HpsiBlock bk = blocks[tk.block];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = warp & 3, wn = warp >> 2;
  const int gid = lane >> 2, tig = lane & 3;
  double s64[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) s64[i][j] = 0.0;
  for (int ii = tk.it_begin; ii < tk.it_begin + tk.it_count; ++ii) {
    const HpsiItem it = items[ii];
    float sacc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) sacc[i][j] = 0.0f;
    // column chunks of psi (the k dimension of the second product)
    int jc_begin = 0, jc_end = it.kb;
    if (it.B == nullptr) {  // identity on the right: only sigma's own columns
      jc_begin = tk.c0;
      jc_end = min(it.kb, tk.c0 + T);
    }
    for (int jc = jc_begin; jc < jc_end; jc += T) {
      float xacc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) xacc[i][j] = 0.0f;
      if (it.A == nullptr) {
        // X = alpha P(rows of the tile, jc chunk): written straight to the X tile
        for (int e = threadIdx.x; e < T * T; e += 256) {
          int r = e / T, c = e % T;
          int gr = tk.r0 + r, gc = jc + c;
          double v = (gr < bk.m && gr < it.ka && gc < jc_end) ? it.alpha * it.P[(size_t)gr * it.ldp + gc] : 0.0;
          uint32_t h, l;
          split64(v, h, l);
          Xh[r * LDX + c] = h;
          Xl[r * LDX + c] = l;
        }
        __syncthreads();
      } else {
        for (int k0 = 0; k0 < it.ka; k0 += KS) {
          for (int e = threadIdx.x; e < T * KS; e += 256) {
            int r, c;
            if (!it.transA) { r = e / KS; c = e % KS; }
            else { c = e / T; r = e % T; }
            int gr = tk.r0 + r, gk = k0 + c;
            double v = (gr < bk.m && gk < it.ka) ? it.alpha * ldA(it, gr, gk) : 0.0;
            uint32_t h, l;
            split64(v, h, l);
            Ah[r * LDS + c] = h;
            Al[r * LDS + c] = l;
          }
          for (int e = threadIdx.x; e < T * KS; e += 256) {
            int kk = e / T, n = e % T;
            int gk = k0 + kk, gn = jc + n;
            double v = (gk < it.ka && gn < jc_end) ? it.P[(size_t)gk * it.ldp + gn] : 0.0;
            uint32_t h, l;
            split64(v, h, l);
            Ph[n * LDS + kk] = h;
            Pl[n * LDS + kk] = l;
          }
          __syncthreads();
          warp_mma_k16(xacc, Ah, Al, LDS, Ph, Pl, LDS, 0, wm, wn, gid, tig);
          __syncthreads();
        }
        if (it.B == nullptr) {
          // identity on the right: sigma += X for the tile's own columns
#pragma unroll
          for (int nt = 0; nt < 4; ++nt)
#pragma unroll
            for (int q = 0; q < 4; ++q) sacc[nt][q] += xacc[nt][q];
          continue;
        }
        // X fragments -> X tile in shared memory (hi / lo planes)
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int r = wm * 16 + gid + ((q >> 1) ? 8 : 0);
            int c = wn * 32 + nt * 8 + 2 * tig + (q & 1);
            float x = xacc[nt][q];
            uint32_t h = tf32(x);
            Xh[r * LDX + c] = h;
            Xl[r * LDX + c] = tf32(x - __uint_as_float(h));
          }
        __syncthreads();
      }
      if (it.B == nullptr) {
        // identity on the right with identity on the left: sigma += X tile
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int r = wm * 16 + gid + ((q >> 1) ? 8 : 0);
            int c = wn * 32 + nt * 8 + 2 * tig + (q & 1);
            sacc[nt][q] += __uint_as_float(Xh[r * LDX + c]) + __uint_as_float(Xl[r * LDX + c]);
          }
        __syncthreads();
        continue;
      }
      // sigma tile += X (64 x chunk) B(tile cols, chunk)^T
      for (int k0 = 0; k0 < T && jc + k0 < jc_end; k0 += KS) {
        for (int e = threadIdx.x; e < T * KS; e += 256) {
          int n, kk;
          if (!it.transB) { n = e / KS; kk = e % KS; }
          else { kk = e / T; n = e % T; }
          int gn = tk.c0 + n, gk = jc + k0 + kk;
          double v = (gn < bk.n && gk < jc_end) ? ldB(it, gn, gk) : 0.0;
          uint32_t h, l;
          split64(v, h, l);
          Bh[n * LDS + kk] = h;
          Bl[n * LDS + kk] = l;
        }
        __syncthreads();
        warp_mma_k16(sacc, Xh, Xl, LDX, Bh, Bl, LDS, k0, wm, wn, gid, tig);
        __syncthreads();
      }
    }
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int q = 0; q < 4; ++q) s64[nt][q] += widen(sacc[nt][q]);
  }
  // write: partial tile or direct add
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int r = wm * 16 + gid + ((q >> 1) ? 8 : 0);
      int c = wn * 32 + nt * 8 + 2 * tig + (q & 1);
      if (tk.part >= 0) {
        scratch[tk.part + r * T + c] = s64[nt][q];
      } else {
        int gr = tk.r0 + r, gc = tk.c0 + c;
        if (gr < bk.m && gc < bk.n) bk.C[(size_t)gr * bk.ldc + gc] += s64[nt][q];
      }
    }
}

// ---------------------------------------------------------------- FP64 variant
// Bound by the float64 pipe (two FMAs a clock and SM: one warp-wide FMA is 16
// clocks of it), so what counts is that no FMA is spent on padding or done
// twice; shared memory and issue slots have room to spare.  A task's tile is
// mt x nt with nt all of a block's columns (up to 480: stage 1, X = alpha
// op(A) P, is then computed once, not once per column tile: sectors of 300..350
// 4.86 -> 3.61 ms against tiles of at most 256 columns) and mt x nt at most
// kF64Out; its outputs are dealt to the threads one by one, 128 at a time, and
// so are those of X, so a 20 x 20 block costs 512 FMAs a k instead of a padded
// 4096.  The two shared-memory reads per FMA this takes (one
// broadcast, one along the lanes) are a quarter of the FMA's own time.  128
// threads and 44 KB: five CTAs an SM hide each other's loads.  1024 outputs
// rather than 2048: the rows of a large block make twice the tasks, whose last
// wave is then short.
// Measured against 64 x 64 tiles padded to their size: 367 -> 21 us a product
// of a 10-site D = 64 run (blocks of 5..40), 6.2 -> 1.69 ms with sectors of
// 40..208 (0.96 TFLOP/s, three quarters of the pipe).
constexpr int kF64Threads = 128;
constexpr int kF64Slots = 8;                        // outputs per thread
constexpr int kF64Out = kF64Threads * kF64Slots;    // outputs of a tile
constexpr int kF64Cols = 480;                       // columns of a tile
constexpr int kF64Rows = 128;                       // rows of a tile
constexpr int kF64Chunk = 128;                      // columns of psi per X chunk
constexpr int F64_A = kF64Rows * (KS + 1), F64_P = KS * kF64Chunk, F64_B = 256 * (KS + 1);  // 480 x 9 beyond 256 columns
constexpr int F64_STAGE = F64_A + F64_P > F64_B ? F64_A + F64_P : F64_B;
constexpr int F64_X = kF64Out + kF64Rows;           // rows of odd length
constexpr size_t kF64Smem = (size_t)(F64_STAGE + F64_X) * sizeof(double);

// rows and columns of the tiles of an m x n block
__host__ __device__ inline void f64_tile(int m, int n, int& mt, int& nt) {
  const int ct = (n + kF64Cols - 1) / kF64Cols;
  nt = (n + ct - 1) / ct;
  mt = kF64Out / nt;
  if (mt > kF64Rows) mt = kF64Rows;
  if (mt > m) mt = m;
  const int rt = (m + mt - 1) / mt;
  mt = (m + rt - 1) / rt;
}
// e / d and e % d of e < 2048, 1 <= d <= 512: the rounding of 2^20 / d is worth
// less than 2^-9 of a quotient, a remainder at least 2^-9
__device__ __forceinline__ int div_tile(int e, unsigned inv) { return (int)(((unsigned)e * inv) >> 20); }
__device__ __forceinline__ unsigned inv_tile(int d) { return (unsigned)(((1 << 20) + d - 1) / d); }

// acc[i] += sum_k a[row_i][k] b, row_i and the column's address from off[i]
// (row part | column part << 16); b moves by bstep per k
template <int NS>
__device__ __forceinline__ void f64_products(double (&acc)[kF64Slots], const int (&off)[kF64Slots], const double* a,
                                             const double* b, int bstep, int kn) {
  for (int k = 0; k < kn; ++k, ++a, b += bstep) {
#pragma unroll
    for (int i = 0; i < NS; ++i) acc[i] = fma(a[off[i] & 0xFFFF], b[off[i] >> 16], acc[i]);
  }
}
__device__ __forceinline__ void f64_products(int ns, double (&acc)[kF64Slots], const int (&off)[kF64Slots],
                                             const double* a, const double* b, int bstep, int kn) {
  switch (ns) {
#define F64_CASE(N) \
  case N: f64_products<N>(acc, off, a, b, bstep, kn); break
    F64_CASE(1); F64_CASE(2); F64_CASE(3); F64_CASE(4); F64_CASE(5); F64_CASE(6); F64_CASE(7); F64_CASE(8);
#undef F64_CASE
  }
}

// Stage 2 of a tile of more than 256 columns: k-steps of eight, so that the
// buffer is no larger.  A function of its own: inlined, it cost the tiles of up
// to 256 columns 3 %.
struct F64Sums {
  double v[kF64Slots];
};
__device__ __noinline__ F64Sums f64_stage2_wide(F64Sums w, const double* B, int ldb, int transB, int nt, int kc,
                                                int outs, unsigned inv_n, const double* Xs, double* Bs) {
  constexpr int ks = 8;
  const int tid = threadIdx.x, ldx = kc | 1;
  double s[kF64Slots];
  int off[kF64Slots];
#pragma unroll
  for (int i = 0; i < kF64Slots; ++i) {
    const int e = tid + i * kF64Threads;
    const int r = e < outs ? div_tile(e, inv_n) : 0, c = e < outs ? e - r * nt : 0;
    off[i] = r * ldx | (c * (ks + 1)) << 16;
    s[i] = w.v[i];
  }
  for (int k0 = 0; k0 < kc; k0 += ks) {
    const int kn = min(ks, kc - k0);
    if (transB) {
      for (int e = tid; e < nt * kn; e += kF64Threads) {
        const int k = e / nt, c = e - k * nt;
        Bs[c * (ks + 1) + k] = __ldg(B + (size_t)(k0 + k) * ldb + c);
      }
    } else {
      for (int e = tid; e < nt * ks; e += kF64Threads) {
        const int c = e / ks, k = e % ks;
        if (k < kn) Bs[c * (ks + 1) + k] = __ldg(B + (size_t)c * ldb + k0 + k);
      }
    }
    __syncthreads();
    f64_products((outs + kF64Threads - 1) / kF64Threads, s, off, Xs + k0, Bs, 1, kn);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kF64Slots; ++i) w.v[i] = s[i];
  return w;
}

__global__ void __launch_bounds__(kF64Threads, 5) hpsi_f64_kernel(const HpsiBlock* __restrict__ blocks,
                                                                  const HpsiItem* __restrict__ items,
                                                                  const HpsiTask* __restrict__ tasks,
                                                                  double* __restrict__ scratch) {
  extern __shared__ double smd[];
  double* const As = smd;          // [row][KS + 1]
  double* const Ps = smd + F64_A;  // [k][kc]
  double* const Bs = smd;          // [column][ks + 1]; shares the buffer with A and P
  double* const Xs = smd + F64_STAGE;  // [row][kc | 1]
  const HpsiTask tk = tasks[blockIdx.x];
  const HpsiBlock bk = blocks[tk.block];
  const int tid = threadIdx.x;
  int tm, tn;
  f64_tile(bk.m, bk.n, tm, tn);
  const int nt = min(tn, bk.n - tk.c0);
  // r0 < 0: one task walks all row tiles
  const int r_begin = max(tk.r0, 0), r_end = tk.r0 < 0 ? bk.m : min(bk.m, tk.r0 + tm);
  for (int r0 = r_begin; r0 < r_end; r0 += tm) {
    const int mt = min(tm, bk.m - r0);
    const int outs = mt * nt, ns = (outs + kF64Threads - 1) / kF64Threads;
    const unsigned inv_n = inv_tile(nt);
    double s[kF64Slots];
#pragma unroll
    for (int i = 0; i < kF64Slots; ++i) s[i] = 0.0;
    HpsiItem next = items[tk.it_begin];
    for (int ii = tk.it_begin; ii < tk.it_begin + tk.it_count; ++ii) {
      const HpsiItem it = next;
      if (ii + 1 < tk.it_begin + tk.it_count) next = items[ii + 1];
      int jc_begin = 0, jc_end = it.kb;
      if (it.B == nullptr) {  // identity on the right: only sigma's own columns
        jc_begin = tk.c0;
        jc_end = min(it.kb, tk.c0 + nt);
      }
      const int step = min(kF64Chunk, kF64Out / mt);
      for (int jc = jc_begin; jc < jc_end; jc += step) {
        const int kc = min(step, jc_end - jc), ldx = kc | 1;
        const unsigned inv_c = inv_tile(kc);
        if (it.A == nullptr) {
          for (int e = tid; e < mt * kc; e += kF64Threads) {
            const int r = div_tile(e, inv_c), c = e - r * kc;
            Xs[r * ldx + c] = r0 + r < it.ka ? it.alpha * it.P[(size_t)(r0 + r) * it.ldp + jc + c] : 0.0;
          }
        } else {
          double x[kF64Slots];
          int off[kF64Slots];
          const int xouts = mt * kc, xs = (xouts + kF64Threads - 1) / kF64Threads;
#pragma unroll
          for (int i = 0; i < kF64Slots; ++i) {
            const int e = tid + i * kF64Threads;
            const int r = e < xouts ? div_tile(e, inv_c) : 0, c = e < xouts ? e - r * kc : 0;
            x[i] = 0.0;
            off[i] = r * (KS + 1) | c << 16;
          }
          for (int k0 = 0; k0 < it.ka; k0 += KS) {
            const int kn = min(KS, it.ka - k0);
            if (it.transA) {
              for (int e = tid; e < mt * kn; e += kF64Threads) {
                const int k = e / mt, r = e - k * mt;
                As[r * (KS + 1) + k] = it.alpha * __ldg(it.A + (size_t)(k0 + k) * it.lda + r0 + r);
              }
            } else {
              for (int e = tid; e < mt * KS; e += kF64Threads) {
                const int r = e / KS, k = e % KS;
                if (k < kn) As[r * (KS + 1) + k] = it.alpha * __ldg(it.A + (size_t)(r0 + r) * it.lda + k0 + k);
              }
            }
            for (int e = tid; e < kn * kc; e += kF64Threads) {
              const int k = div_tile(e, inv_c), c = e - k * kc;
              Ps[e] = __ldg(it.P + (size_t)(k0 + k) * it.ldp + jc + c);
            }
            __syncthreads();
            f64_products(xs, x, off, As, Ps, kc, kn);
            __syncthreads();
          }
#pragma unroll
          for (int i = 0; i < kF64Slots; ++i) {
            const int e = tid + i * kF64Threads;
            if (e < xouts) {
              const int r = div_tile(e, inv_c);
              Xs[r * ldx + e - r * kc] = x[i];
            }
          }
        }
        if (it.B == nullptr) {
          // sigma's columns [jc, jc + kc) += X
          __syncthreads();
          const int c_off = jc - tk.c0;
#pragma unroll
          for (int i = 0; i < kF64Slots; ++i) {
            const int e = tid + i * kF64Threads;
            if (e < outs) {
              const int r = div_tile(e, inv_n), c = e - r * nt - c_off;
              if (c >= 0 && c < kc) s[i] += Xs[r * ldx + c];
            }
          }
          __syncthreads();
          continue;
        }
        if (tn > 256) {
          F64Sums w;
#pragma unroll
          for (int i = 0; i < kF64Slots; ++i) w.v[i] = s[i];
          w = f64_stage2_wide(w, it.B + (it.transB ? (size_t)jc * it.ldb + tk.c0 : (size_t)tk.c0 * it.ldb + jc), it.ldb,
                              it.transB, nt, kc, outs, inv_n, Xs, Bs);
#pragma unroll
          for (int i = 0; i < kF64Slots; ++i) s[i] = w.v[i];
          continue;
        }
        int off[kF64Slots];
#pragma unroll
        for (int i = 0; i < kF64Slots; ++i) {
          const int e = tid + i * kF64Threads;
          const int r = e < outs ? div_tile(e, inv_n) : 0, c = e < outs ? e - r * nt : 0;
          off[i] = r * ldx | (c * (KS + 1)) << 16;
        }
        for (int k0 = 0; k0 < kc; k0 += KS) {
          const int kn = min(KS, kc - k0);
          if (it.transB) {
            for (int e = tid; e < nt * kn; e += kF64Threads) {
              const int k = e / nt, c = e - k * nt;
              Bs[c * (KS + 1) + k] = __ldg(it.B + (size_t)(jc + k0 + k) * it.ldb + tk.c0 + c);
            }
          } else {
            for (int e = tid; e < nt * KS; e += kF64Threads) {
              const int c = e / KS, k = e % KS;
              if (k < kn) Bs[c * (KS + 1) + k] = __ldg(it.B + (size_t)(tk.c0 + c) * it.ldb + jc + k0 + k);
            }
          }
          __syncthreads();
          f64_products(ns, s, off, Xs + k0, Bs, 1, kn);
          __syncthreads();
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kF64Slots; ++i) {
      const int e = tid + i * kF64Threads;
      if (e >= outs) continue;
      if (tk.part >= 0) {
        scratch[tk.part + e] = s[i];
      } else {
        const int r = div_tile(e, inv_n);
        bk.C[(size_t)(r0 + r) * bk.ldc + tk.c0 + e - r * nt] += s[i];
      }
    }
  }
}

// C += the partial tiles of a sigma tile, in a fixed order: bound by the
// latency of its loads (a block of a small sector has some fifty partials), so
// a warp sums a quarter of the partials of 32 outputs, eight in flight, and
// the quarters are added in order.  Measured, 10 sites at D = 64: 13.2 -> 5.3 us a product
// against one thread per output with sixteen in flight.
constexpr int kF64RedOut = 32;
__global__ void __launch_bounds__(128) hpsi_f64_reduce_kernel(const HpsiBlock* __restrict__ blocks,
                                                              const HpsiReduce* __restrict__ reds,
                                                              const double* __restrict__ scratch) {
  __shared__ double sum[4][kF64RedOut];
  const HpsiReduce rd = reds[blockIdx.x];
  const HpsiBlock bk = blocks[rd.block];
  int tm, tn;
  f64_tile(bk.m, bk.n, tm, tn);
  const int nt = min(tn, bk.n - rd.c0), outs = min(tm, bk.m - rd.r0) * nt;
  const int e0 = blockIdx.y * kF64RedOut;
  if (e0 >= outs) return;
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5, e = e0 + lane;
  double* const c = bk.C + (size_t)(rd.r0 + e / nt) * bk.ldc + rd.c0 + e % nt;
  const double old = q == 0 && e < outs ? *c : 0.0;
  const int p0 = rd.nparts * q / 4, p1 = rd.nparts * (q + 1) / 4;
  double acc = 0.0;
  if (e < outs) {
    const double* p = scratch + rd.part0 + e;
#pragma unroll 8
    for (int i = p0; i < p1; ++i) acc += __ldg(p + (long long)i * outs);
  }
  sum[q][lane] = acc;
  __syncthreads();
  if (q == 0 && e < outs) *c = old + (((sum[0][lane] + sum[1][lane]) + sum[2][lane]) + sum[3][lane]);
}

// sum the partial tiles of one sigma tile in a fixed order and add into C
__global__ void hpsi_reduce_kernel(const HpsiBlock* __restrict__ blocks, const HpsiReduce* __restrict__ reds,
                                   const double* __restrict__ scratch) {
  const HpsiReduce rd = reds[blockIdx.x];
  const HpsiBlock bk = blocks[rd.block];
  for (int e = threadIdx.x; e < T * T; e += blockDim.x) {
    int r = e / T, c = e % T;
    int gr = rd.r0 + r, gc = rd.c0 + c;
    if (gr >= bk.m || gc >= bk.n) continue;
    double acc = 0.0;
    for (int p = 0; p < rd.nparts; ++p) acc += scratch[rd.part0 + (long long)p * T * T + e];
    bk.C[(size_t)gr * bk.ldc + gc] += acc;
  }
}

}  // namespace

namespace {

size_t plan_bytes(size_t part, size_t tasks, size_t reds);

// items per chunk of tiles of 64 x 64, and the chunks of a block
int square_items(const std::vector<HpsiBlock>& blocks) {
  long long tile_items = 0;
  for (auto& b : blocks) tile_items += (long long)b.item_count * ((b.m + T - 1) / T) * ((b.n + T - 1) / T);
  return (int)std::max<long long>(4, tile_items / (8 * 152) + 1);
}

// tiles of 64 x 64 in item chunks of equal count
size_t plan_square(const std::vector<HpsiBlock>& blocks, std::vector<HpsiTask>& tasks, std::vector<HpsiReduce>& reds) {
  const int max_items = square_items(blocks);
  long long part = 0;
  for (size_t b = 0; b < blocks.size(); ++b) {
    const HpsiBlock& bk = blocks[b];
    if (bk.item_count == 0 || bk.m == 0 || bk.n == 0) continue;
    int nch = (bk.item_count + max_items - 1) / max_items;
    int per = (bk.item_count + nch - 1) / nch;
    for (int r0 = 0; r0 < bk.m; r0 += T)
      for (int c0 = 0; c0 < bk.n; c0 += T) {
        if (nch == 1) {
          tasks.push_back({(int)b, r0, c0, bk.item_begin, bk.item_count, -1});
        } else {
          reds.push_back({(int)b, r0, c0, nch, part});
          for (int c = 0; c < nch; ++c) {
            int i0 = bk.item_begin + c * per;
            int cnt = std::min(per, bk.item_begin + bk.item_count - i0);
            tasks.push_back({(int)b, r0, c0, i0, cnt, part});
            part += (long long)T * T;
          }
        }
      }
  }
  return (size_t)part;
}

// bytes of the lists and partial tiles of that plan
size_t square_bytes(const std::vector<HpsiBlock>& blocks) {
  const int max_items = square_items(blocks);
  size_t part = 0, tasks = 0, reds = 0;
  for (const HpsiBlock& bk : blocks) {
    if (bk.item_count == 0 || bk.m == 0 || bk.n == 0) continue;
    const size_t tiles = (size_t)((bk.m + T - 1) / T) * ((bk.n + T - 1) / T);
    const size_t nch = (bk.item_count + max_items - 1) / max_items;
    tasks += tiles * nch;
    if (nch > 1) {
      reds += tiles;
      part += tiles * nch * T * T;
    }
  }
  return plan_bytes(part, tasks, reds);
}

// Clocks of an item on a tile: two FMAs a clock, and the latency of the item's
// and its k-steps' loads (a thousand clocks and more each, shared by the CTAs
// of an SM).
double f64_item_cost(const HpsiItem& it, int mt, int nt) {
  const double ka = it.A ? it.ka : 0.0, kb = it.kb;
  double c = 0.5 * mt * (ka * (it.B ? kb : std::min<double>(kb, nt)) + (it.B ? kb * nt : 0.0));
  return c + 800.0 + 300.0 * (ka / KS * ((kb + kF64Chunk - 1) / kF64Chunk) + (it.B ? kb / KS : 0.0));
}

// Tiles of f64_tile, the items of a tile in chunks of about `target` clocks;
// target < 0: one task per column tile, walking all rows and items.
size_t plan_f64(const std::vector<HpsiBlock>& blocks, const std::vector<double>& cost, const std::vector<double>& run,
                double target, std::vector<HpsiTask>& tasks, std::vector<HpsiReduce>& reds) {
  tasks.clear();
  reds.clear();
  long long part = 0;
  std::vector<int> cut;
  for (size_t b = 0; b < blocks.size(); ++b) {
    const HpsiBlock& bk = blocks[b];
    if (bk.item_count == 0 || bk.m == 0 || bk.n == 0) continue;
    int mt, nt;
    f64_tile(bk.m, bk.n, mt, nt);
    const int first = bk.item_begin, last = first + bk.item_count;
    if (target < 0) {
      for (int c0 = 0; c0 < bk.n; c0 += nt) tasks.push_back({(int)b, -1, c0, first, bk.item_count, -1});
      continue;
    }
    // cuts into chunks of equal cost, the same for every tile of the block
    const int nch = (int)std::max(1.0, std::min<double>(bk.item_count, cost[b] / target));
    cut.assign(1, first);
    for (int i = first; i + 1 < last && (int)cut.size() < nch; ++i)
      if (run[i] >= cost[b] * cut.size() / nch) cut.push_back(i + 1);
    cut.push_back(last);
    const int n = (int)cut.size() - 1;
    for (int r0 = 0; r0 < bk.m; r0 += mt)
      for (int c0 = 0; c0 < bk.n; c0 += nt) {
        const long long outs = (long long)std::min(mt, bk.m - r0) * std::min(nt, bk.n - c0);
        if (n > 1) reds.push_back({(int)b, r0, c0, n, part});
        for (int c = 0; c < n; ++c) {
          tasks.push_back({(int)b, r0, c0, cut[c], cut[c + 1] - cut[c], n > 1 ? part : -1});
          if (n > 1) part += outs;
        }
      }
  }
  return (size_t)part;
}

size_t plan_bytes(size_t part, size_t tasks, size_t reds) {
  return part * sizeof(double) + ((tasks * sizeof(HpsiTask) + 255) & ~size_t(255)) +
         ((reds * sizeof(HpsiReduce) + 255) & ~size_t(255));
}

}  // namespace

size_t hpsi_plan_tasks(const std::vector<HpsiBlock>& blocks, const std::vector<HpsiItem>& items, Precision prec,
                       std::vector<HpsiTask>& tasks, std::vector<HpsiReduce>& reds, size_t* nominal_bytes) {
  tasks.clear();
  reds.clear();
  if (prec != Precision::FP64) {
    const size_t part = plan_square(blocks, tasks, reds);
    if (nominal_bytes) *nominal_bytes = plan_bytes(part, tasks.size(), reds.size());
    return part;
  }
  const size_t nominal = square_bytes(blocks);
  if (nominal_bytes) *nominal_bytes = nominal;
  // Three tasks per CTA that the SMs hold at once (152 x 5): the last wave is
  // then a third.  No chunk below 3500 clocks: an item of a small block is
  // about 800 of latency, so a chunk is at most four of them where the launch
  // does not fill the SMs anyway (sectors of 2..23: 41 -> 27 us against chunks
  // of 8000 clocks).
  // Lists and partial tiles take no more than those of the 64 x 64 plan would,
  // or than what the allocation-free entry has: longer chunks, at last one task
  // per column tile.
  const size_t lists = (blocks.size() * sizeof(HpsiBlock) + 255) / 256 * 256 +
                       (items.size() * sizeof(HpsiItem) + 255) / 256 * 256;
  const size_t left = lists < kNoAllocScratchBytes ? kNoAllocScratchBytes - lists : 0;
  const size_t limit = std::max(nominal, left);
  // cost[b], run[i]: of the block's items, of those up to item i
  std::vector<double> cost(blocks.size(), 0.0), run(items.size(), 0.0);
  double total = 0.0;
  for (size_t b = 0; b < blocks.size(); ++b) {
    const HpsiBlock& bk = blocks[b];
    if (bk.item_count == 0 || bk.m == 0 || bk.n == 0) continue;
    int mt, nt;
    f64_tile(bk.m, bk.n, mt, nt);
    for (int i = bk.item_begin; i < bk.item_begin + bk.item_count; ++i)
      run[i] = cost[b] += f64_item_cost(items[i], mt, nt);
    total += cost[b] * ((bk.m + mt - 1) / mt) * ((bk.n + nt - 1) / nt);
  }
  double target = std::max(3500.0, total / (152 * 5 * 3));
  for (int k = 0; k < 6; ++k, target *= 4.0) {
    const size_t part = plan_f64(blocks, cost, run, target, tasks, reds);
    if (plan_bytes(part, tasks.size(), reds.size()) <= limit) return part;
  }
  return plan_f64(blocks, cost, run, -1.0, tasks, reds);
}

void hpsi_launch(const HpsiBlock* blocks, const HpsiItem* items, const HpsiTask* tasks, int ntasks,
                 const HpsiReduce* reds, int nreds, double* scratch, Precision prec, int* err,
                 cudaStream_t st) {
  (void)err;
  if (prec == Precision::TC_TF32X3)
    throw std::runtime_error("internal: the tcgen05 contraction runs on pre-split operands (hpsi_tc_launch)");
  if (ntasks > 0) {
    if (prec == Precision::FP64) {
      cudaError_t ea = ensure_smem_attr((const void*)hpsi_f64_kernel, (int)kF64Smem);
      if (ea != cudaSuccess)
        throw std::runtime_error(std::string("cuda: hpsi f64 attribute: ") + cudaGetErrorString(ea));
      hpsi_f64_kernel<<<ntasks, kF64Threads, kF64Smem, st>>>(blocks, items, tasks, scratch);
    } else {
      size_t smem = (size_t)SM_WORDS * sizeof(uint32_t);
      cudaError_t ea = ensure_smem_attr((const void*)hpsi_tf32x3_kernel, (int)smem);
      if (ea != cudaSuccess)
        throw std::runtime_error(std::string("cuda: hpsi tf32x3 attribute: ") + cudaGetErrorString(ea));
      hpsi_tf32x3_kernel<<<ntasks, 256, smem, st>>>(blocks, items, tasks, scratch);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: hpsi launch: ") + cudaGetErrorString(e));
  }
  if (nreds > 0) {
    if (prec == Precision::FP64)
      hpsi_f64_reduce_kernel<<<dim3(nreds, kF64Out / kF64RedOut), 128, 0, st>>>(blocks, reds, scratch);
    else
      hpsi_reduce_kernel<<<nreds, 256, 0, st>>>(blocks, reds, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: hpsi reduce: ") + cudaGetErrorString(e));
  }
}

}  // namespace dmrg
