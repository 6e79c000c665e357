// Kernels of the batched float64 eigensolver (eigh.cuh).
//
// GB300 has two float64 FMAs a clock and SM and float64 divisions and square
// roots of some hundred clocks, so the chains of rotations of Jacobi and QL
// iterations are what a solver has to avoid; a cyclic Jacobi on groups of CTAs
// (this file's predecessor) spent 13 n^3 FMAs and 10 n group barriers on a
// matrix.  Here a matrix costs n^3 FMAs and n barriers of tridiagonalisation,
// n^3 FMAs of reflectors, and GEMMs on the tensor cores.  Measured, the 13
// density matrices of 9..601 of a decimation: 184 ms before; now 10.6 ms, of
// which the tridiagonalisation 5.5, the reflectors 2.8, the merges 1.9 with
// their products, the small matrices and leaves 0.4; the largest error of the
// eigenvectors 3e-12 -> 4e-13.
#include <algorithm>
#include <cmath>
#include <stdexcept>
#include <string>
#include <type_traits>

#include "eigh.cuh"
#include "kattr.hpp"

namespace dmrg {

namespace {

constexpr double kEps = 2.220446049250313e-16;

void check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: ") + what + ": " + cudaGetErrorString(e));
}
void check_attr(const void* f, size_t smem, const char* what) {
  const cudaError_t e = ensure_smem_attr(f, (int)smem);
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: ") + what + " attribute: " + cudaGetErrorString(e));
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
  return x;
}
// sum over the CTA in a fixed order; red holds blockDim / 32 values and is
// free again after the next barrier of the caller
__device__ __forceinline__ double block_sum(double x, double* red) {
  x = warp_sum(x);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  const int nw = blockDim.x >> 5;  // four
  x = red[0];
  for (int i = 1; i < nw; ++i) x += red[i];
  return x;
}
__device__ __forceinline__ unsigned block_max(unsigned x, unsigned* red) {
  x = __reduce_max_sync(0xffffffffu, x);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  const int nw = blockDim.x >> 5;
  x = (int)(threadIdx.x & 31) < nw ? red[threadIdx.x & 31] : 0u;
  return __reduce_max_sync(0xffffffffu, x);
}
// high word of |x| for the largest entry; non-finite entries do not count
__device__ __forceinline__ unsigned magnitude(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7FFFFFFFu;
  return h < 0x7FF00000u ? h : 0u;
}
// 2^e of a largest entry's high word, and 2^-e: both normal numbers
__device__ __forceinline__ void power_of_two(unsigned hi, double& s, double& inv) {
  const int be = min((int)(hi >> 20), 2045);
  s = be < 1 ? 1.0 : __hiloint2double(be << 20, 0);
  inv = be < 1 ? 1.0 : __hiloint2double((2046 - be) << 20, 0);
}
// order of eigenvalues: NaN below everything, ties by index
__device__ __forceinline__ double sort_key(double x) { return x == x ? x : -INFINITY; }

// ---------------------------------------------------------------- small matrices
constexpr int SMALL_THREADS = 128;
constexpr int SMALL_LD = kEighSmall + 1;
constexpr int kMaxSweeps = 30;

struct SmallShared {
  double a[kEighSmall * SMALL_LD];
  double v[kEighSmall * SMALL_LD];  // row p: eigenvector p
  double cs[kEighSmall / 2], sn[kEighSmall / 2];
  int pp[kEighSmall / 2], qq[kEighSmall / 2];
  double red[SMALL_THREADS / 32];
  int rotations;
};

// Parallel cyclic Jacobi (round-robin pairing) of the n x n matrix in sh.a:
// sh.a ends diagonal, sh.v holds the eigenvectors as rows.  A round rotates
// n / 2 disjoint pairs; the matrix is updated as 2 x 2 blocks of pairs i <= j,
// each result stored at both symmetric positions.  A pair is skipped when its
// entry is negligible next to both diagonal entries or below 1e-16 ||A||_F,
// the rounding noise of a product that formed the matrix; the iteration stops
// after a sweep without rotations.
// Bound by latency: a warp-wide float64 operation holds its quarter of an SM
// for 64 clocks, whatever the number of its lanes, and a division or a square
// root is some ten of them.  A rotation only has to be orthogonal to float64
// rounding, its angle may be approximate: the tangent is computed in float32,
// and the cosine from it by one third-order step on a float32 inverse square
// root (an entry of 1 shrinks to 1e-7 instead of 1e-17, which a later sweep
// finishes); the updates are dealt to all four warps in pieces of eight
// operations.
__device__ void jacobi_small(SmallShared& sh, int n) {
  const int tid = threadIdx.x;
  const int np = (n + 1) & ~1, h = np / 2, M = np - 1;
  double fro = 0.0;
  for (int e = tid; e < n * n; e += SMALL_THREADS) {
    const int r = e / n, c = e - r * n;
    const double x = sh.a[r * SMALL_LD + c];
    fro += x * x;
    sh.v[r * SMALL_LD + c] = r == c ? 1.0 : 0.0;
  }
  if (n & 1)
    for (int r = tid; r < n; r += SMALL_THREADS) sh.v[r * SMALL_LD + n] = 0.0;
  // the largest entries are about one (of the whole matrix, for a leaf of it)
  const double floor_abs = fmax(1e-16 * sqrt(block_sum(fro, sh.red)), 1e-30);
  // blocks (i, j), i <= j, of this thread: the row-major upper triangle
  const int nb = h * (h + 1) / 2;
  int bi[2], bj[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int e = tid + u * SMALL_THREADS, i = 0;
    if (e < nb)
      while (e >= h - i) e -= h - i, ++i;
    bi[u] = i;
    bj[u] = tid + u * SMALL_THREADS < nb ? i + e : -1;
  }
  // the first thread without a block (of the last round of them) takes the
  // first piece of the eigenvectors; columns n and beyond are scratch
  const int hc = (n + 1) / 2, v0 = (tid + SMALL_THREADS - nb % SMALL_THREADS) % SMALL_THREADS;
  __syncthreads();
  for (int sweep = 0; sweep < kMaxSweeps && n > 1; ++sweep) {
    if (tid == 0) sh.rotations = 0;
    __syncwarp();
    for (int round = 0; round < M; ++round) {
      if (tid < h) {
        // pairs of the round: (round, M) and (round + i, round - i) mod M
        int p = round + tid, q = round - tid;
        if (p >= M) p -= M;
        if (q < 0) q += M;
        if (tid == 0) q = M;
        if (p > q) {
          const int t = p;
          p = q;
          q = t;
        }
        double c = 1.0, s = 0.0;
        if (q < n) {
          const double apq = sh.a[p * SMALL_LD + q], app = sh.a[p * SMALL_LD + p], aqq = sh.a[q * SMALL_LD + q];
          const float f = (float)apq;
          // an entry below the rounding of a hundredth of both diagonal entries is left
          if (fabs(apq) > floor_abs && !(fabsf(f) < 1.1e-18f * fminf(fabsf((float)app), fabsf((float)aqq)))) {
            const float th = __fdividef((float)(aqq - app), 2.0f * f);
            const float t = copysignf(__frcp_rn(fabsf(th) + __fsqrt_rn(fmaf(th, th, 1.0f))), th);
            const double td = t, u = fma(td, td, 1.0), y = (double)rsqrtf(fmaf(t, t, 1.0f));
            const double r = fma(-u, y * y, 1.0);  // about 2^-22: the next term of the series is below 2^-64
            c = fma(y * r, fma(0.375, r, 0.5), y);
            s = td * c;
            if (s != 0.0) atomicAdd(&sh.rotations, 1);
          }
        }
        sh.cs[tid] = c;
        sh.sn[tid] = s;
        sh.pp[tid] = p;
        sh.qq[tid] = q;
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int i = bi[u], j = bj[u];
        if (j < 0) continue;
        const double ci = sh.cs[i], si = sh.sn[i], cj = sh.cs[j], sj = sh.sn[j];
        if (si == 0.0 && sj == 0.0) continue;
        const int p = sh.pp[i], q = sh.qq[i], r = sh.pp[j], t = sh.qq[j];
        const bool qv = q < n, tv = t < n;
        double* const a = sh.a;
        const double x00 = a[p * SMALL_LD + r], x01 = tv ? a[p * SMALL_LD + t] : 0.0;
        const double x10 = qv ? a[q * SMALL_LD + r] : 0.0, x11 = qv && tv ? a[q * SMALL_LD + t] : 0.0;
        const double y00 = ci * x00 - si * x10, y01 = ci * x01 - si * x11;
        const double y10 = si * x00 + ci * x10, y11 = si * x01 + ci * x11;
        const double n00 = cj * y00 - sj * y01, n01 = sj * y00 + cj * y01;
        const double n10 = cj * y10 - sj * y11, n11 = sj * y10 + cj * y11;
        a[p * SMALL_LD + r] = a[r * SMALL_LD + p] = n00;
        if (tv) a[p * SMALL_LD + t] = a[t * SMALL_LD + p] = n01;
        if (qv && i != j) a[q * SMALL_LD + r] = a[r * SMALL_LD + q] = n10;
        if (qv && tv) a[q * SMALL_LD + t] = a[t * SMALL_LD + q] = n11;
      }
      // two columns of the eigenvector rows p, q of pair i
      for (int e = v0; e < h * hc; e += SMALL_THREADS) {
        const int i = e / hc, k = 2 * (e - i * hc);
        const double s = sh.sn[i];
        if (s == 0.0) continue;
        const double c = sh.cs[i];
        double *vp = sh.v + sh.pp[i] * SMALL_LD + k, *vq = sh.v + sh.qq[i] * SMALL_LD + k;
        const double x0 = vp[0], y0 = vq[0], x1 = vp[1], y1 = vq[1];
        vp[0] = c * x0 - s * y0;
        vq[0] = s * x0 + c * y0;
        vp[1] = c * x1 - s * y1;
        vq[1] = s * x1 + c * y1;
      }
      __syncthreads();
    }
    const bool done = sh.rotations == 0;
    __syncthreads();
    if (done) break;
  }
}
// rank of diagonal entry i among the n, descending or ascending
__device__ __forceinline__ int small_rank(const SmallShared& sh, int n, int i, bool descending) {
  const double di = sort_key(sh.a[i * SMALL_LD + i]);
  int rank = 0;
  for (int j = 0; j < n; ++j) {
    const double dj = sort_key(sh.a[j * SMALL_LD + j]);
    rank += (descending ? dj > di : dj < di) || (dj == di && j < i);
  }
  return rank;
}
// sign that makes the first of the largest components (up to 1e-12) positive;
// x(k) for k < n, called by a whole warp
template <class F>
__device__ __forceinline__ double positive_largest(int n, F x) {
  const int lane = threadIdx.x & 31;
  double m = 0.0;
  for (int k = lane; k < n; k += 32) m = fmax(m, fabs(x(k)));
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, d));
  for (int k0 = 0; k0 < n; k0 += 32) {
    const double v = k0 + lane < n ? x(k0 + lane) : 0.0;
    const unsigned hit = __ballot_sync(0xffffffffu, k0 + lane < n && fabs(v) >= m - 1e-12);
    if (hit) return __shfl_sync(0xffffffffu, v, __ffs(hit) - 1) < 0.0 ? -1.0 : 1.0;
  }
  return 1.0;
}

__global__ void __launch_bounds__(SMALL_THREADS) eigh_small_kernel(const EighTask* __restrict__ tasks) {
  __shared__ SmallShared sh;
  __shared__ unsigned ured[SMALL_THREADS / 32];
  const EighTask tk = tasks[blockIdx.x];
  const int n = tk.n, tid = threadIdx.x;
  unsigned mx = 0u;
  for (int e = tid; e < n * n; e += SMALL_THREADS) mx = max(mx, magnitude(tk.A[e]));
  double scale, inv;
  power_of_two(block_max(mx, ured), scale, inv);
  for (int e = tid; e < n * n; e += SMALL_THREADS) sh.a[e / n * SMALL_LD + e % n] = tk.A[e] * inv;
  __syncthreads();
  jacobi_small(sh, n);
  const int lane = tid & 31;
  for (int i = tid >> 5; i < n; i += SMALL_THREADS / 32) {
    const int rank = small_rank(sh, n, i, true);
    const double* src = sh.v + i * SMALL_LD;
    const double sg = positive_largest(n, [&](int k) { return src[k]; });
    if (lane == 0) tk.w[rank] = sh.a[i * SMALL_LD + i] * scale;
    if (lane < n) tk.V[rank * n + lane] = sg * src[lane];
  }
}

// ---------------------------------------------------------------- tridiagonalisation
// T = Q^T A Q by reflectors H_k = 1 - c v v^T, the trailing matrix kept whole
// and updated at once by - v w^T - w v^T.  The CTAs of a group hold its rows
// interleaved, in shared memory where they fit.  All of them know the next row,
// v and w, so a step needs one exchange: every CTA publishes its part of
// p = A v and the owner of the next row that row before its update, and with
// both everyone forms w, the updated row and the next reflector, the same in
// every CTA.  The update of a row and its product with the next v are one pass.
// What is published carries its step in the same 16 bytes, so a reader waits
// for the value itself and the exchange is one trip through L2 in place of a
// barrier (fence, arrival, poll) and a read.  A step takes the place of the one
// two before: everyone who reads a step publishes in the next (a CTA with
// nothing to publish there leaves without reading), and everyone waits for all
// of that before it publishes once more.
// Bound by the float64 pipe (a warp-wide operation holds a quarter of an SM
// for 64 clocks): three FMAs per entry, n^3 in all, and what every CTA repeats,
// so a CTA is four warps, one per quarter, each with up to four rows in flight
// that share the reads of v and w and one tree of sums (always four left the
// quarters unevenly loaded: 11600 clocks of the pass of the largest of 13
// matrices, 4800 of them FMAs of an even load).  The rest of a step is a
// chain of latencies: v is not scaled (no division before the pass, the
// division for c runs while the others' parts travel), the norm comes from an
// inverse square root.  Measured, the tridiagonalisation of 13 matrices of 9..601:
// 7.7 ms with sixteen warps and a barrier, 6.7 with four, 6.1 without it, 5.5 with
// the rows dealt evenly.
constexpr int TRI_WARPS = 4, TRI_THREADS = 32 * TRI_WARPS, TRI_ROWS = 4;
constexpr size_t kTriSmem = 220 * 1024;

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned x;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
  return x;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// a value and the step it belongs to, written and read as one
__device__ __forceinline__ void publish(double2* at, double x, long long step) {
  asm volatile("{\n.reg .b128 v;\nmov.b128 v, {%1, %2};\nst.relaxed.gpu.global.b128 [%0], v;\n}\n" ::"l"(at),
               "l"(__double_as_longlong(x)), "l"(step)
               : "memory");
}
__device__ __forceinline__ bool published(const double2* at, long long step, double& x) {
  long long v, t;
  asm volatile("{\n.reg .b128 v;\nld.relaxed.gpu.global.b128 v, [%2];\nmov.b128 {%0, %1}, v;\n}\n"
               : "=l"(v), "=l"(t)
               : "l"(at)
               : "memory");
  x = __longlong_as_double(v);
  return t == step;
}
// waits until `target` CTAs have arrived; false when the wait ran out (a bound
// of 0: when it was not over at its first probe)
__device__ bool group_barrier(unsigned* bar, unsigned target, int* ok_s, unsigned long long wait_ns) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    const unsigned long long t0 = global_ns();
    const int spin = wait_ns > 0 ? 256 : 1;
    for (int probe = 0; ld_acquire(bar) < target; ++probe) {
      if (probe >= spin && global_ns() - t0 >= wait_ns) {
        *ok_s = 0;
        break;
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *ok_s != 0;
}

template <bool kSmem>
__device__ void tridiag_one(const DcMatrix& mt, const DcArrays& ar, int mat, int me, double* sm, double* red,
                            int* ok_s, int* err, unsigned long long wait_ns) {
  const int n = mt.n, g = mt.g, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* const A = mt.A;
  double* v = sm;                // row k of the trailing matrix, then the reflector
  double* vo = v + n;            // the reflector before, and its w
  double* x = vo + n;            // the next row
  double* const wo = x + n;
  double* const pl = wo + n;     // p
  double* const rows = pl + n;   // kSmem: row lr g + me at lr n
  double* const first = red + 2 * TRI_WARPS;  // x[k + 1], by parity of k
  const int nloc = (n - me + g - 1) / g, scribe = (n - 1) % g;
  auto row = [&](int lr) { return kSmem ? rows + (size_t)lr * n : A + (size_t)(lr * g + me) * n; };
  // own rows, and the largest entry of all: one barrier
  unsigned mx = 0u;
  unsigned* const peak = (unsigned*)mt.peak;
  double s = 0.0, scale, inv;
  for (int lr = warp; lr < nloc; lr += TRI_WARPS) {
    const double* src = A + (size_t)(lr * g + me) * n;
#pragma unroll 8
    for (int j = lane; j < n; j += 32) {
      const double y = __ldcg(src + j);
      mx = max(mx, magnitude(y));
      if (kSmem) rows[(size_t)lr * n + j] = y;
    }
  }
  if (tid == 0) *ok_s = 1;
  for (int j = tid; j < n; j += TRI_THREADS) {
    v[j] = __ldcg(A + j);
    vo[j] = wo[j] = 0.0;
  }
  mx = block_max(mx, (unsigned*)red);
  if (g > 1) {
    if (tid == 0) __stcg(peak + me, mx);
    if (!group_barrier(mt.bar, g, ok_s, wait_ns)) goto fail;
    mx = 0u;
    for (int i = tid; i < g; i += TRI_THREADS) mx = max(mx, __ldcg(peak + i));
    mx = block_max(mx, (unsigned*)red);
  }
  power_of_two(mx, scale, inv);
  if (me == scribe && tid == 0) ar.scale[mat] = scale;
  for (int lr = warp; lr < nloc; lr += TRI_WARPS) {
    // row 0 goes on in v alone; in global memory the scribe puts its reflector
    // there without waiting for anyone
    if (!kSmem && lr == 0 && me == 0) continue;
    double* const a = row(lr);
    for (int j = lane; j < n; j += 32) a[j] *= inv;
  }
  for (int j = tid; j < n; j += TRI_THREADS) {
    const double y = v[j] * inv;
    v[j] = y;
    if (j == 1) first[0] = y;
    if (j > 1) s = fma(y, y, s);
  }
  __syncthreads();  // red is free again
  for (int k = 0; k + 1 < n; ++k) {
    // the reflector of v[k + 1 ...], s = this thread's part of |v[k + 2 ...]|^2
    s = block_sum(s, red);
    const double alpha = first[k & 1];
    // a tail below 1e-30 of the matrix is left out (its squares would lose
    // digits to underflow, and H its orthogonality)
    const bool reflect = s > 1e-60;
    const double s2 = fma(alpha, alpha, s), norm = reflect ? s2 * rsqrt(s2) : 0.0;
    const double v1 = alpha + copysign(norm, alpha);
    if (tid == 0) v[k + 1] = v1;
    if (me == scribe && tid == 0) {
      ar.d[mt.off + k] = v[k];
      ar.e[mt.off + k] = reflect ? -copysign(norm, alpha) : alpha;
    }
    __syncthreads();
    const long long step = k + 1;
    double2* const pub = (double2*)mt.xch + (size_t)(k & 1) * 2 * n;  // p, then the next row
    const int live = k < me ? 0 : (k - me) / g + 1;                   // first local row beyond k
    if (g > 1 && live < nloc && live * g + me == k + 1) {
      // the next row before this step's update (its last update is below)
      const double* a = row(live);
      const double vi = vo[k + 1], wi = wo[k + 1];
      // rows in global memory: the scribe overwrites this one with a reflector,
      // after what this CTA stored there
      if (!kSmem) __threadfence();
      for (int j = k + 1 + tid; j < n; j += TRI_THREADS) publish(pub + n + j, fma(-wi, vo[j], fma(-vi, wo[j], a[j])), step);
      __syncthreads();
    }
    // rows of a warp at a time: as many as deal the rows evenly to the warps
    const int active = nloc - live, rounds = (active + TRI_ROWS * TRI_WARPS - 1) / (TRI_ROWS * TRI_WARPS);
    auto update = [&](auto per_warp) {
      constexpr int R = decltype(per_warp)::value;
      for (int lr = live + R * warp; lr < nloc; lr += R * TRI_WARPS) {
        double* a[R];
        double vi[R], wi[R], acc[R];
        bool keep[R];  // the next row is the scribe's from here on
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int q = min(lr + r, nloc - 1);
          a[r] = row(q);
          keep[r] = g == 1 || q * g + me != k + 1;
          vi[r] = vo[q * g + me];
          wi[r] = wo[q * g + me];
          acc[r] = 0.0;
        }
        const int rows_here = min(R, nloc - lr);
        if (rows_here == R) {
#pragma unroll 2
          for (int j = k + 1 + lane; j < n; j += 32) {
            const double vj = vo[j], wj = wo[j], nj = v[j];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              const double y = fma(-wi[r], vj, fma(-vi[r], wj, a[r][j]));
              if (kSmem || keep[r]) a[r][j] = y;
              acc[r] = fma(y, nj, acc[r]);
            }
          }
        } else {
          for (int j = k + 1 + lane; j < n; j += 32) {
            const double vj = vo[j], wj = wo[j], nj = v[j];
#pragma unroll
            for (int r = 0; r < R - 1; ++r)
              if (r < rows_here) {
                const double y = fma(-wi[r], vj, fma(-vi[r], wj, a[r][j]));
                if (kSmem || keep[r]) a[r][j] = y;
                acc[r] = fma(y, nj, acc[r]);
              }
          }
        }
        // the sums in one tree: the first lane of each quarter (half, for two
        // rows; warp, for one) ends with a row's
        double t = acc[0];
        int r = 0, lanes = 32;
        if constexpr (R > 2) {
          const bool up = lane & 16, odd = lane & 8;
          const double a3 = R > 3 ? acc[R - 1] : 0.0;
          double t0 = up ? acc[2] : acc[0], t1 = up ? a3 : acc[1];
          t0 += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[2], 16);
          t1 += __shfl_xor_sync(0xffffffffu, up ? acc[1] : a3, 16);
          t = odd ? t1 : t0;
          t += __shfl_xor_sync(0xffffffffu, odd ? t0 : t1, 8);
          r = lane >> 3;
          lanes = 8;
        } else if constexpr (R == 2) {
          const bool up = lane & 16;
          t = up ? acc[1] : acc[0];
          t += __shfl_xor_sync(0xffffffffu, up ? acc[0] : acc[1], 16);
          t += __shfl_xor_sync(0xffffffffu, t, 8);
          r = lane >> 4;
          lanes = 16;
        } else {
          t += __shfl_xor_sync(0xffffffffu, t, 16);
          t += __shfl_xor_sync(0xffffffffu, t, 8);
        }
#pragma unroll
        for (int d = 4; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
        if ((lane & (lanes - 1)) == 0 && r < rows_here) {
          if (g > 1) publish(pub + (lr + r) * g + me, t, step);
          else pl[lr + r] = t;
        }
      }
    };
    switch (rounds > 0 ? (active + TRI_WARPS * rounds - 1) / (TRI_WARPS * rounds) : 0) {
      case 1: update(std::integral_constant<int, 1>()); break;
      case 2: update(std::integral_constant<int, 2>()); break;
      case 3: update(std::integral_constant<int, 3>()); break;
      case 4: update(std::integral_constant<int, 4>()); break;
    }
    // row k of the matrix is done: it keeps the reflector
    if (me == scribe)
      for (int j = k + 1 + tid; j < n; j += TRI_THREADS) A[(size_t)k * n + j] = v[j];
    // no rows after the next one: nothing to publish any more, so nobody would
    // wait for this CTA's reading
    if (me != scribe && (nloc - 1) * g + me <= k + 1) return;
    const double c = reflect ? 1.0 / fma(fabs(alpha), norm, s2) : 0.0;
    if (me == scribe && tid == 0) ar.tau[mt.off + k] = c;
    // w = c p - c^2 (p v) / 2 v, and the next row
    double pv = 0.0;
    if (g > 1) {
      const unsigned long long t0 = global_ns();
      constexpr int BATCH = 3;
      for (int j0 = k + 1 + tid; j0 < n; j0 += BATCH * TRI_THREADS) {
        double p[BATCH], y[BATCH];
        bool all;
        for (int probe = 0;; ++probe) {
          all = true;
#pragma unroll
          for (int q = 0; q < BATCH; ++q) {
            const int j = j0 + q * TRI_THREADS;
            if (j < n) {
              const bool a1 = published(pub + j, step, p[q]), a2 = published(pub + n + j, step, y[q]);
              all = all && a1 && a2;
            }
          }
          if (all) break;
          if (wait_ns == 0 || ((probe & 63) == 63 && global_ns() - t0 >= wait_ns)) break;
        }
        if (!all) {
          *ok_s = 0;
          break;
        }
#pragma unroll
        for (int q = 0; q < BATCH; ++q) {
          const int j = j0 + q * TRI_THREADS;
          if (j < n) {
            pl[j] = p[q];
            x[j] = y[q];
            pv = fma(p[q], v[j], pv);
          }
        }
      }
    } else {
      __syncthreads();
      const double* a = row(k + 1);
      for (int j = k + 1 + tid; j < n; j += TRI_THREADS) {
        x[j] = a[j];
        pv = fma(pl[j], v[j], pv);
      }
    }
    if (!kSmem) __threadfence();
    pv = 0.5 * c * c * block_sum(pv, red + TRI_WARPS);
    if (!*(volatile int*)ok_s) goto fail;
    const double w1 = fma(-pv, v1, c * pl[k + 1]);
    s = 0.0;
    for (int j = k + 1 + tid; j < n; j += TRI_THREADS) {
      const double vj = v[j], w = fma(-pv, vj, c * pl[j]);
      wo[j] = w;
      const double y = fma(-w1, vj, fma(-v1, w, x[j]));
      x[j] = y;
      if (j == k + 2) first[(k + 1) & 1] = y;
      if (j > k + 2) s = fma(y, y, s);  // for the next reflector
    }
    // x is the next v; the barrier of the next sum makes it visible
    double* const free_row = vo;
    vo = v;
    v = x;
    x = free_row;
  }
  __syncthreads();
  if (me == scribe && tid == 0) {
    ar.d[mt.off + n - 1] = v[n - 1];
    ar.e[mt.off + n - 1] = 0.0;
    ar.tau[mt.off + n - 1] = 0.0;
  }
  return;
fail:
  if (tid == 0) atomicExch(err, 1);
}

__global__ void __launch_bounds__(TRI_THREADS, 1) tridiag_kernel(const DcMatrix* __restrict__ mats, int m0, int count,
                                                                 DcArrays ar, int* __restrict__ err,
                                                                 unsigned long long wait_ns) {
  extern __shared__ double sm[];
  __shared__ double red[2 * TRI_WARPS + 2];
  __shared__ int ok_s;
  // CTA b belongs to the last matrix whose first CTA is at most b
  int lo = m0, hi = m0 + count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (mats[mid].cta0 <= (int)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const DcMatrix mt = mats[lo];
  const int me = (int)blockIdx.x - mt.cta0;
  // five vectors beyond shared memory (n > 5632)
  if (5 * (size_t)mt.n * sizeof(double) > kTriSmem)
    tridiag_one<false>(mt, ar, lo, me, ar.wide + (size_t)blockIdx.x * 5 * mt.n, red, &ok_s, err, wait_ns);
  else if (mt.rows_in_smem) tridiag_one<true>(mt, ar, lo, me, sm, red, &ok_s, err, wait_ns);
  else tridiag_one<false>(mt, ar, lo, me, sm, red, &ok_s, err, wait_ns);
}

// ---------------------------------------------------------------- divide and conquer
// Leaves: T with every |e| of a cut taken off the two diagonal entries beside
// it, [lo, lo + n1) solved by Jacobi.
__global__ void __launch_bounds__(SMALL_THREADS) dc_leaf_kernel(const DcMatrix* __restrict__ mats,
                                                                const DcNode* __restrict__ nodes, DcArrays ar) {
  __shared__ SmallShared sh;
  const DcNode nd = nodes[blockIdx.x];
  const DcMatrix& mt = mats[nd.mat];
  const int n = nd.n1, tid = threadIdx.x;
  const double *d = ar.d + nd.off, *e = ar.e + nd.off;
  for (int t = tid; t < n * n; t += SMALL_THREADS) {
    const int r = t / n, c = t - r * n;
    double y = 0.0;
    if (r == c) {
      y = d[r];
      if (r == 0 && nd.lo > 0) y -= fabs(e[-1]);
      if (r == n - 1 && nd.lo + n < mt.n) y -= fabs(e[r]);
    } else if (r - c == 1 || c - r == 1) {
      y = e[min(r, c)];
    }
    sh.a[r * SMALL_LD + c] = y;
  }
  __syncthreads();
  jacobi_small(sh, n);
  const int lane = tid & 31;
  for (int i = tid >> 5; i < n; i += SMALL_THREADS / 32) {
    const int rank = small_rank(sh, n, i, false);
    if (lane == 0) ar.val[nd.off + rank] = sh.a[i * SMALL_LD + i];
    if (lane < n) mt.B[0][(size_t)(nd.lo + rank) * mt.n + nd.lo + lane] = sh.v[i * SMALL_LD + lane];
  }
}

constexpr int PREP_THREADS = 256;
constexpr int kPrepMax = 8000;  // 28 B a position of shared memory
// A merge, D + rho z z^T: the poles sorted, those with a negligible z and one
// of each pair that a rotation decouples set aside (deflation, to 8 eps of the
// largest entry).  The walk along the sorted poles is a serial chain of one
// thread (about 100 clocks a pole, no division unless a pair is rotated).
__global__ void __launch_bounds__(PREP_THREADS) dc_prepare_kernel(const DcMatrix* __restrict__ mats,
                                                                  const DcNode* __restrict__ nodes, int level,
                                                                  int largest, DcArrays ar) {
  extern __shared__ double sm[];
  __shared__ double red[PREP_THREADS / 32];
  const DcNode nd = nodes[blockIdx.x];
  const DcMatrix& mt = mats[nd.mat];
  const int n1 = nd.n1, N = n1 + nd.n2, tid = threadIdx.x;
  // (a merge beyond shared memory: in the flat array)
  double* const val = largest > kPrepMax ? ar.wide + 4 * (size_t)nd.off : sm;
  double* const ds = val + N;
  double* const zs = ds + N;
  int* const ps = (int*)(zs + N);
  const double e = ar.e[nd.off + n1 - 1];
  const double rho = 2.0 * fabs(e), sgn = e < 0.0 ? -1.0 : 1.0;
  const double* V = mt.B[level & 1] + (size_t)nd.lo * mt.n + nd.lo;
  for (int i = tid; i < N; i += PREP_THREADS) {
    val[i] = ar.val[nd.off + i];
    ps[i] = i;
    ds[i] = zs[i] = 0.0;
  }
  __syncthreads();
  double big = 0.0;
  for (int i = tid; i < N; i += PREP_THREADS) {
    const double di = sort_key(val[i]);
    const bool first = i < n1;
    // entries of the other child in front of this one
    int lo = first ? n1 : 0, hi = first ? N : n1;
    const int base = lo;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      const double dm = sort_key(val[mid]);
      if (first ? dm < di : dm <= di) lo = mid + 1;
      else hi = mid;
    }
    const int r = (first ? i : i - n1) + (lo - base);
    const double z = 0.7071067811865476 * (first ? 1.0 : sgn) * V[(size_t)i * mt.n + (first ? n1 - 1 : n1)];
    ds[r] = val[i];
    zs[r] = z;
    ps[r] = i;
    big = fmax(big, fmax(fabs(val[i]), fabs(z)));
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) big = fmax(big, __shfl_xor_sync(0xffffffffu, big, d));
  if ((tid & 31) == 0) red[tid >> 5] = big;
  __syncthreads();
  if (tid != 0) return;
  for (int i = 1; i < PREP_THREADS / 32; ++i) big = fmax(big, red[i]);
  const double tol = 8.0 * kEps * big;
  double *dl = ar.dl + nd.off, *zl = ar.zl + nd.off;
  int* pos = ar.pos + nd.off;
  DcRot* rot = ar.rot + nd.off;
  int K = 0, nrot = 0, back = N, pj = -1;
  double dp = 0.0, zp = 0.0;
  int pp = 0;
  for (int r = 0; r < N; ++r) {
    const double dr = ds[r], zr = zs[r];
    const int pr = ps[r];
    if (rho * fabs(zr) <= tol) {
      --back;
      dl[back] = dr;
      pos[back] = pr;
      continue;
    }
    double dn = dr, zn = zr;
    if (pj >= 0) {
      const double q = fma(zp, zp, zr * zr);
      if (fabs((dr - dp) * (zp * zr)) <= tol * q) {
        const double len = sqrt(q), c = zr / len, s = -zp / len;
        rot[nrot++] = DcRot{pp, pr, c, s};
        --back;
        dl[back] = fma(dp, c * c, dr * (s * s));
        pos[back] = pp;
        dn = fma(dp, s * s, dr * (c * c));
        zn = len;
      } else {
        dl[K] = dp;
        zl[K] = zp;
        pos[K] = pp;
        ++K;
      }
    }
    pj = r;
    dp = dn;
    zp = zn;
    pp = pr;
  }
  if (pj >= 0) {
    dl[K] = dp;
    zl[K] = zp;
    pos[K] = pp;
    ++K;
  }
  ar.count[2 * nd.off] = K;
  ar.count[2 * nd.off + 1] = nrot;
  ar.rho[nd.off] = rho;
}

// the node and item of flat index t (items of the nodes one after another)
__device__ __forceinline__ bool dc_item(const DcNode* nodes, int count, int t, DcNode& nd, int& item) {
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (nodes[mid].first <= t) lo = mid;
    else hi = mid - 1;
  }
  nd = nodes[lo];
  item = t - nd.first;
  return item < nd.n1 + nd.n2;
}

// Root j of 1 / rho + sum z_i^2 / (d_i - x) in (d_j, d_{j+1}), one warp.  The
// unknown is mu = x - (the nearer pole); every step replaces the sums left and
// right of x by r + s / (d_j - x) and r' + s' / (d_{j+1} - x) of the same value
// and slope and solves the quadratic, with a bracket around the root.
__global__ void __launch_bounds__(256) dc_roots_kernel(const DcNode* __restrict__ nodes, int count, int positions,
                                                       DcArrays ar) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= positions) return;
  DcNode nd;
  int j;
  if (!dc_item(nodes, count, t, nd, j)) return;
  const int K = ar.count[2 * nd.off];
  if (j >= K) return;
  const double *d = ar.dl + nd.off, *z = ar.zl + nd.off;
  const double rho = ar.rho[nd.off], irho = 1.0 / rho;
  const bool last = j == K - 1;
  const double dj = d[j];
  double lo, hi, mu, org = dj;
  int o = j;
  if (last) {
    double s = 0.0;
    for (int i = lane; i < K; i += 32) s = fma(z[i], z[i], s);
    hi = rho * warp_sum(s);
    lo = 0.0;
    mu = hi;
  } else {
    const double gap = d[j + 1] - dj, mid = 0.5 * gap;
    double s = 0.0;
    for (int i = lane; i < K; i += 32) s += z[i] * z[i] / ((d[i] - dj) - mid);
    s = irho + warp_sum(s);
    if (s >= 0.0) {
      lo = 0.0;
      hi = mid;
      mu = mid;
    } else {
      o = j + 1;
      org = d[j + 1];
      lo = -mid;
      hi = 0.0;
      mu = -mid;
    }
  }
  const double pj = dj - org, pn = last ? 0.0 : d[j + 1] - org;
  for (int it = 0; it < 80; ++it) {
    double psi = 0.0, dpsi = 0.0, phi = 0.0, dphi = 0.0;
    for (int i = lane; i < K; i += 32) {
      const double q = 1.0 / ((d[i] - org) - mu), zq = z[i] * q, f = zq * z[i], df = zq * zq;
      if (i <= j) {
        psi += f;
        dpsi += df;
      } else {
        phi += f;
        dphi += df;
      }
    }
    psi = warp_sum(psi);
    dpsi = warp_sum(dpsi);
    if (!last) {
      phi = warp_sum(phi);
      dphi = warp_sum(dphi);
    }
    const double f = irho + psi + phi;
    if (!(fabs(f) > 8.0 * kEps * (irho + fabs(psi) + fabs(phi)))) break;  // also NaN
    if (f >= 0.0) hi = mu;
    else lo = mu;
    const double D1 = pj - mu;
    double eta;
    const double s1 = dpsi * D1 * D1;
    if (last) {
      const double c = irho + psi - dpsi * D1;
      eta = D1 + s1 / c;
    } else {
      const double D2 = pn - mu, s2 = dphi * D2 * D2;
      const double c = irho + (psi - dpsi * D1) + (phi - dphi * D2);
      const double a = c * (D1 + D2) + s1 + s2, b = D1 * D2 * f;
      const double r = sqrt(fabs(a * a - 4.0 * b * c));
      eta = a <= 0.0 ? (c == 0.0 ? b / a : (a - r) / (2.0 * c)) : 2.0 * b / (a + r);
    }
    double next = mu + eta;
    if (!(next > lo && next < hi)) {
      // not inside: the middle of the bracket, geometric where it starts at the pole
      next = lo == 0.0 ? hi * 0.0625 : hi == 0.0 ? lo * 0.0625 : 0.5 * (lo + hi);
      if (!(next > lo && next < hi)) break;
    } else if (fabs(eta) <= 0.5 * kEps * fabs(next)) {
      mu = next;
      break;
    }
    mu = next;
  }
  if (lane == 0) {
    ar.mu[nd.off + j] = mu;
    ar.org[nd.off + j] = o;
  }
}

// z of the update whose roots are exactly the computed ones (their products of
// differences), the eigenvalues in ascending order and where each one came from
__global__ void __launch_bounds__(256) dc_update_kernel(const DcNode* __restrict__ nodes, int count, int positions,
                                                        DcArrays ar) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= positions) return;
  DcNode nd;
  int i;
  if (!dc_item(nodes, count, t, nd, i)) return;
  const int N = nd.n1 + nd.n2, K = ar.count[2 * nd.off];
  const double *d = ar.dl + nd.off, *mu = ar.mu + nd.off;
  const int* org = ar.org + nd.off;
  const double di = d[i];
  if (i < K) {
    double p = 1.0;
    for (int j = lane; j < K; j += 32) {
      const double x = (d[org[j]] - di) + mu[j];
      p *= j == i ? x : x / (d[j] - di);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) p *= __shfl_xor_sync(0xffffffffu, p, s);
    if (lane == 0) ar.zhat[nd.off + i] = copysign(sqrt(fabs(p)), ar.zl[nd.off + i]);
  }
  const double vi = i < K ? d[org[i]] + mu[i] : di, key = sort_key(vi);
  int rank = 0;
  for (int j = lane; j < N; j += 32) {
    const double vj = sort_key(j < K ? d[org[j]] + mu[j] : d[j]);
    rank += vj < key || (vj == key && j < i);
  }
  rank = __reduce_add_sync(0xffffffffu, rank);
  if (lane == 0) {
    ar.val[nd.off + rank] = vi;
    ar.inv[nd.off + rank] = i;
  }
}

// 1 / norm of the vector z_i / (d_i - x_j) of root j
__global__ void __launch_bounds__(256) dc_norm_kernel(const DcNode* __restrict__ nodes, int count, int positions,
                                                      DcArrays ar) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= positions) return;
  DcNode nd;
  int j;
  if (!dc_item(nodes, count, t, nd, j)) return;
  const int K = ar.count[2 * nd.off];
  if (j >= K) return;
  const double *d = ar.dl + nd.off, *zh = ar.zhat + nd.off;
  const double org = d[ar.org[nd.off + j]], mu = ar.mu[nd.off + j];
  double s = 0.0;
  for (int i = lane; i < K; i += 32) {
    const double u = zh[i] / ((d[i] - org) - mu);
    s = fma(u, u, s);
  }
  s = warp_sum(s);
  if (lane == 0) ar.ninv[nd.off + j] = 1.0 / sqrt(s);
}

// U (DcMatrix::V, the node's diagonal block): row = row of the children's
// eigenvectors, column = rank of the new eigenvalue; then the rotations of the
// deflation, last one first.  CTA: 128 columns of a node.  The nodes are the
// grid's x: a batch of small matrices has more of them than y may count (65535).
constexpr int FILL_COLS = 128;
__global__ void __launch_bounds__(FILL_COLS) dc_fill_kernel(const DcMatrix* __restrict__ mats,
                                                            const DcNode* __restrict__ nodes, DcArrays ar) {
  const DcNode nd = nodes[blockIdx.x];
  const DcMatrix& mt = mats[nd.mat];
  const int N = nd.n1 + nd.n2, K = ar.count[2 * nd.off];
  const int c = blockIdx.y * FILL_COLS + threadIdx.x;
  if (c >= N) return;
  const int j = ar.inv[nd.off + c];
  const double *d = ar.dl + nd.off, *zh = ar.zhat + nd.off;
  const int* pos = ar.pos + nd.off;
  const bool kept = j < K;
  const double org = kept ? d[ar.org[nd.off + j]] : 0.0, mu = kept ? ar.mu[nd.off + j] : 0.0;
  const double ninv = kept ? ar.ninv[nd.off + j] : 0.0;
  double* const U = mt.V + (size_t)nd.lo * mt.n + nd.lo + c;
  const int zn = gridDim.z, i0 = (int)((long long)N * blockIdx.z / zn), i1 = (int)((long long)N * (blockIdx.z + 1) / zn);
#pragma unroll 4
  for (int i = i0; i < i1; ++i) {
    double u = i == j ? 1.0 : 0.0;
    if (kept) u = i < K ? zh[i] * ninv / ((d[i] - org) - mu) : 0.0;
    U[(size_t)pos[i] * mt.n] = u;
  }
}
__global__ void __launch_bounds__(FILL_COLS) dc_rotate_kernel(const DcMatrix* __restrict__ mats,
                                                              const DcNode* __restrict__ nodes, DcArrays ar) {
  const DcNode nd = nodes[blockIdx.x];
  const DcMatrix& mt = mats[nd.mat];
  const int c = blockIdx.y * FILL_COLS + threadIdx.x, nrot = ar.count[2 * nd.off + 1];
  if (c >= nd.n1 + nd.n2) return;
  double* const U = mt.V + (size_t)nd.lo * mt.n + nd.lo + c;
  for (int r = nrot - 1; r >= 0; --r) {
    const DcRot q = ar.rot[nd.off + r];
    double *up = U + (size_t)q.p * mt.n, *uq = U + (size_t)q.q * mt.n;
    const double x = *up, y = *uq;
    *up = q.c * x - q.s * y;
    *uq = q.s * x + q.c * y;
  }
}

// ---------------------------------------------------------------- back transformation
// Eigenvectors of A: reflectors n - 3 ... 0 applied to a row of B (a
// eigenvector of T), one warp per vector, the vector in shared memory.  Bound
// by the float64 pipe (n^2 FMAs a vector; the shared-memory traffic of an FMA
// is a fifth of its time).  Then the sign, and the descending order.
__global__ void __launch_bounds__(128) dc_back_kernel(const DcMatrix* __restrict__ mats, int count, int rows,
                                                      int largest, DcArrays ar) {
  extern __shared__ double sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = blockIdx.x * (blockDim.x >> 5) + warp;
  if (t >= rows) return;
  int lo = 0, hi = count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (mats[mid].off <= t) lo = mid;
    else hi = mid - 1;
  }
  const DcMatrix& mt = mats[lo];
  const int n = mt.n, r = t - mt.off;
  double* const y = sm + (size_t)warp * largest;
  const double* src = mt.B[mt.levels & 1] + (size_t)r * n;
  for (int j = lane; j < n; j += 32) y[j] = src[j];
  __syncwarp();
  for (int k = n - 3; k >= 0; --k) {
    const double tau = __ldg(ar.tau + mt.off + k);
    if (tau == 0.0) continue;
    const double* v = mt.A + (size_t)k * n;
    double s0 = 0.0, s1 = 0.0;
    int j = k + 1 + lane;
    for (; j + 32 < n; j += 64) {
      s0 = fma(__ldg(v + j), y[j], s0);
      s1 = fma(__ldg(v + j + 32), y[j + 32], s1);
    }
    if (j < n) s0 = fma(__ldg(v + j), y[j], s0);
    const double s = -tau * warp_sum(s0 + s1);
#pragma unroll 4
    for (j = k + 1 + lane; j < n; j += 32) y[j] = fma(s, __ldg(v + j), y[j]);
    __syncwarp();  // the next reflector deals the entries to other lanes
  }
  __syncwarp();
  const double sg = positive_largest(n, [&](int k) { return y[k]; });
  double* const out = mt.V + (size_t)(n - 1 - r) * n;
  for (int j = lane; j < n; j += 32) out[j] = sg * y[j];
  if (lane == 0) mt.w[n - 1 - r] = ar.val[t] * ar.scale[lo];
}

}  // namespace

// ---------------------------------------------------------------- host
int dc_levels(int n) {
  int l = 0;
  while ((n + (1 << l) - 1) >> l > kEighLeaf) ++l;
  return l;
}

DcPlan dc_plan(const std::vector<int>& sizes) {
  DcPlan p;
  int off = 0, deepest = 0;
  for (int n : sizes) deepest = std::max(deepest, dc_levels(n));
  p.merges.resize(deepest);
  for (size_t m = 0; m < sizes.size(); ++m) {
    const int L = dc_levels(sizes[m]);
    // blocks at depth `depth`, halved from the whole
    std::vector<int> cut{0, sizes[m]};
    for (int depth = 0; depth <= L; ++depth) {
      std::vector<int> next;
      for (size_t b = 0; b + 1 < cut.size(); ++b) {
        const int lo = cut[b], n = cut[b + 1] - lo, n1 = n / 2;
        if (depth == L) p.leaves.push_back({(int)m, off + lo, lo, n, 0, 0});
        else p.merges[L - 1 - depth].push_back({(int)m, off + lo, lo, n1, n - n1, 0});
        next.push_back(lo);
        next.push_back(lo + n1);
      }
      next.push_back(sizes[m]);
      cut = next;
    }
    off += sizes[m];
  }
  for (auto& level : p.merges) {
    int at = 0;
    for (DcNode& nd : level) {
      nd.first = at;
      at += nd.n1 + nd.n2;
    }
  }
  return p;
}

static size_t tri_bytes(int n, int g, bool rows) {
  return (5 * (size_t)n + (rows ? (size_t)((n + g - 1) / g) * n : 0)) * sizeof(double);
}
bool tridiag_rows_fit(int n, int g) { return tri_bytes(n, g, true) <= kTriSmem; }

size_t tridiag_wide(int n, int total, int ctas) {
  size_t w = 0;
  if (tri_bytes(n, 1, false) > kTriSmem) w = (size_t)ctas * 5 * n;
  if (n > kPrepMax) w = std::max(w, 4 * (size_t)total);
  return w;
}

int tridiag_max_ctas(int sms) {
  check_attr((const void*)tridiag_kernel, kTriSmem, "tridiagonalisation");
  int per = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, tridiag_kernel, TRI_THREADS, kTriSmem) != cudaSuccess) {
    cudaGetLastError();
    per = 0;
  }
  return per * sms;
}

void eigh_small_launch(const EighTask* tasks, int count, cudaStream_t st) {
  if (count <= 0) return;
  eigh_small_kernel<<<count, SMALL_THREADS, 0, st>>>(tasks);
  check_launch("small eigensolver");
}

void tridiag_launch(const DcMatrix* mats, int m0, int count, int ctas, DcArrays ar, int* err,
                    unsigned long long wait_ns, cudaStream_t st) {
  void* args[] = {(void*)&mats, (void*)&m0, (void*)&count, (void*)&ar, (void*)&err, (void*)&wait_ns};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)tridiag_kernel, dim3(ctas), dim3(TRI_THREADS), args,
                                                    kTriSmem, st);
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: tridiagonalisation: ") + cudaGetErrorString(e));
}

void dc_leaves_launch(const DcMatrix* mats, const DcNode* nodes, int count, DcArrays ar, cudaStream_t st) {
  if (count <= 0) return;
  dc_leaf_kernel<<<count, SMALL_THREADS, 0, st>>>(mats, nodes, ar);
  check_launch("tridiagonal leaves");
}

void dc_merge_launch(const DcMatrix* mats, const DcNode* nodes, int count, int positions, int largest, int level,
                     DcArrays ar, cudaStream_t st) {
  if (count <= 0) return;
  const size_t smem = largest > kPrepMax ? 0 : (size_t)largest * (3 * sizeof(double) + sizeof(int));
  check_attr((const void*)dc_prepare_kernel, kPrepMax * (3 * sizeof(double) + sizeof(int)), "merge");
  dc_prepare_kernel<<<count, PREP_THREADS, smem, st>>>(mats, nodes, level, largest, ar);
  const int warps = (positions + 7) / 8;
  dc_roots_kernel<<<warps, 256, 0, st>>>(nodes, count, positions, ar);
  dc_update_kernel<<<warps, 256, 0, st>>>(nodes, count, positions, ar);
  dc_norm_kernel<<<warps, 256, 0, st>>>(nodes, count, positions, ar);
  // a column's entries are dealt over as many CTAs as make about two waves of
  // eight per SM
  const int cols = (largest + FILL_COLS - 1) / FILL_COLS;
  const int parts = std::max(1, std::min({64, (largest + 7) / 8, 2432 / std::max(1, cols * count)}));
  dc_fill_kernel<<<dim3(count, cols, parts), FILL_COLS, 0, st>>>(mats, nodes, ar);
  dc_rotate_kernel<<<dim3(count, cols), FILL_COLS, 0, st>>>(mats, nodes, ar);
  check_launch("merge");
}

void dc_back_launch(const DcMatrix* mats, int count, int rows, int largest, DcArrays ar, cudaStream_t st) {
  if (count <= 0) return;
  // four vectors a CTA (one per quarter of an SM): small enough that the last
  // CTAs, of the smallest matrices, even the SMs out
  const int warps = (int)std::max<size_t>(1, std::min<size_t>(4, (110 * 1024) / ((size_t)largest * sizeof(double))));
  const size_t smem = (size_t)warps * largest * sizeof(double);
  check_attr((const void*)dc_back_kernel, 110 * 1024, "back transformation");
  dc_back_kernel<<<(rows + warps - 1) / warps, 32 * warps, smem, st>>>(mats, count, rows, largest, ar);
  check_launch("back transformation");
}

}  // namespace dmrg
