// CUDA implementation of the device primitives (backend.hpp) for sm_103a.
//
// Kernels:
//   place_kernel        C += sum_s alpha_s op(S_s)            (HBM-bound block copies)
//   gemm_f64_kernel     C += sum_s alpha_s op(A_s) op(B_s)    (FP64 on the FMA pipe: small blocks)
//   gemm_digits_kernel (gemm_digits.cu)                        (FP64 as exact bf16 digit products on tcgen05;
//                       fma_missing_kernel adds what the digits hold less well than FMAs)
//   gemm_tf32x3 (gemm_split.cu)                                (split-FP32 tensor-core path)
//   dots/combine/axpby  vector algebra (FP64, deterministic two-stage reductions); davidson.cu has the
//                       fused steps of an iteration
//   eigh.cu             batched FP64 eigensolver: Jacobi for small matrices, tridiagonalisation on groups of
//                       CTAs and divide and conquer for larger ones
// All kernels are bounded loops over their inputs.  What waits gives up after
// the backend's wait bound (2 s by default) and sets an error flag: the CTA
// groups of the tridiagonalisation for one another, the roles of a CTA of the
// digit GEMM and (within its cluster) of the tcgen05 contraction.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <stdexcept>
#include <string>
#include <vector>

#include "backend.hpp"
#include "davidson.cuh"
#include "eigh.cuh"
#include "gemm_digits.cuh"
#include "gemm_split.cuh"
#include "hpsi_fused.cuh"
#include "hpsi_tc.cuh"
#include "jacobi_plan.hpp"

namespace dmrg {

#define CK(x)                                                                          \
  do {                                                                                 \
    cudaError_t e_ = (x);                                                              \
    if (e_ != cudaSuccess)                                                             \
      throw std::runtime_error(std::string("cuda: ") + #x + ": " + cudaGetErrorString(e_)); \
  } while (0)

// ------------------------------------------------------------------ place
struct PlaceTile {
  int group, r0, c0, pad;
};

__global__ void place_kernel(const PlaceGroup* __restrict__ groups, const PlaceSeg* __restrict__ segs,
                             const PlaceTile* __restrict__ tiles) {
  const PlaceTile t = tiles[blockIdx.x];
  const PlaceGroup g = groups[t.group];
  // 32 x 32 tile, 256 threads: 4 rows per thread
  const int c = t.c0 + (threadIdx.x & 31);
  const int rb = t.r0 + (threadIdx.x >> 5);
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  if (c < g.cols) {
    for (int s = g.seg_begin; s < g.seg_begin + g.seg_count; ++s) {
      const PlaceSeg sg = segs[s];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int r = rb + 8 * i;
        if (r >= g.rows) break;
        double v;
        if (sg.src == nullptr) v = (r == c) ? 1.0 : 0.0;
        else v = sg.trans ? sg.src[(size_t)c * sg.ld + r] : sg.src[(size_t)r * sg.ld + c];
        acc[i] += sg.alpha * v;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r = rb + 8 * i;
      if (r >= g.rows) break;
      g.dst[(size_t)r * g.ld + c] += acc[i];
    }
  }
}

// ------------------------------------------------------------------ FP64 GEMM
struct GemmTile {
  int group, r0, c0, pad;
};

constexpr int kTM = 64, kTN = 64, kTK = 16;

__device__ __forceinline__ void gemm_f64_step(const double (*As)[kTM + 1], const double (*Bs)[kTN + 1], int kk,
                                              int tx, int ty, double (&acc)[4][4]) {
  double a[4], b[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
  for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
}

__global__ void __launch_bounds__(256) gemm_f64_kernel(const GemmGroup* __restrict__ groups,
                                                       const GemmSeg* __restrict__ segs,
                                                       const GemmTile* __restrict__ tiles) {
  __shared__ double As[kTK][kTM + 1];
  __shared__ double Bs[kTK][kTN + 1];
  const GemmTile t = tiles[blockIdx.x];
  const GemmGroup g = groups[t.group];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int s = g.seg_begin; s < g.seg_begin + g.seg_count; ++s) {
    const GemmSeg sg = segs[s];
    for (int k0 = 0; k0 < sg.k; k0 += kTK) {
      // A tile (kTM x kTK) -> As[kk][i], scaled by alpha
      for (int e = threadIdx.x; e < kTM * kTK; e += 256) {
        int i, kk;
        if (!sg.transA) { i = e / kTK; kk = e % kTK; }
        else { kk = e / kTM; i = e % kTM; }
        int gi = t.r0 + i, gk = k0 + kk;
        double v = 0.0;
        if (gi < g.m && gk < sg.k)
          v = sg.transA ? sg.A[(size_t)gk * sg.lda + gi] : sg.A[(size_t)gi * sg.lda + gk];
        As[kk][i] = sg.alpha * v;
      }
      for (int e = threadIdx.x; e < kTN * kTK; e += 256) {
        int j, kk;
        if (!sg.transB) { kk = e / kTN; j = e % kTN; }
        else { j = e / kTK; kk = e % kTK; }
        int gj = t.c0 + j, gk = k0 + kk;
        double v = 0.0;
        if (gj < g.n && gk < sg.k)
          v = sg.transB ? sg.B[(size_t)gj * sg.ldb + gk] : sg.B[(size_t)gk * sg.ldb + gj];
        Bs[kk][j] = v;
      }
      __syncthreads();
      // a ragged last step (k = 1 outer products, k tails) runs only its valid kk
      const int kn = min(kTK, sg.k - k0);
      if (kn == kTK) {
#pragma unroll
        for (int kk = 0; kk < kTK; ++kk) gemm_f64_step(As, Bs, kk, tx, ty, acc);
      } else {
        for (int kk = 0; kk < kn; ++kk) gemm_f64_step(As, Bs, kk, tx, ty, acc);
      }
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int gi = t.r0 + ty + 16 * i;
    if (gi >= g.m) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int gj = t.c0 + tx + 16 * j;
      if (gj < g.n) g.C[(size_t)gi * g.ldc + gj] += acc[i][j];
    }
  }
}

// ------------------------------------------------------------------ vectors
constexpr int kRedBlocks = 152;  // one partial per SM for the reductions

__global__ void dots_partial(const double* __restrict__ V, int m, size_t len, size_t ld,
                             const double* __restrict__ x, double* __restrict__ part) {
  // blockIdx.y = vector index, blockIdx.x = chunk
  __shared__ double sh[256];
  const int i = blockIdx.y;
  double s = 0.0;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < len;
       t += (size_t)gridDim.x * blockDim.x)
    s = fma(V[(size_t)i * ld + t], x[t], s);
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)i * gridDim.x + blockIdx.x] = sh[0];
}

__global__ void dots_final(const double* __restrict__ part, int nparts, double* __restrict__ out) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int t = threadIdx.x; t < nparts; t += blockDim.x) s += part[(size_t)blockIdx.x * nparts + t];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = sh[0];
}

__global__ void combine_kernel(double* __restrict__ y, double beta, const double* __restrict__ V,
                               int m, size_t len, size_t ld, const double* __restrict__ c) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < len;
       t += (size_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int i = 0; i < m; ++i) s = fma(c[i], V[(size_t)i * ld + t], s);
    y[t] = (beta == 0.0) ? s : fma(beta, y[t], s);
  }
}

__global__ void axpby_kernel(double* __restrict__ y, double a, const double* __restrict__ x, double b,
                             size_t len) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < len;
       t += (size_t)gridDim.x * blockDim.x)
    y[t] = (a == 0.0) ? b * x[t] : fma(a, y[t], b * x[t]);
}

__global__ void precond_kernel(double* __restrict__ y, const double* __restrict__ x,
                               const double* __restrict__ d, double e, size_t len) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < len;
       t += (size_t)gridDim.x * blockDim.x) {
    double den = d[t] - e;
    if (fabs(den) < 1e-8) den = den < 0 ? -1e-8 : 1e-8;
    y[t] = x[t] / den;
  }
}

// ------------------------------------------------------------------ pinned memory
// Page-locked blocks that outlive a backend: the host entries make one backend
// per call, and allocating and freeing its staging memory took 0.3 to 0.4 ms
// of each.  A block belongs to one backend between get and put (which comes
// after the backend's stream is idle); at most kPinnedKept bytes wait for the
// next one, more is freed.  Portable and mapped, so any device may use it.
class PinnedPool {
 public:
  static PinnedPool& get() {
    static PinnedPool* p = new PinnedPool;  // never destroyed: the driver may be gone before it
    return *p;
  }
  void* take(size_t bytes, size_t* capacity) {
    {
      std::lock_guard<std::mutex> lock(mu_);
      auto it = free_.lower_bound(bytes);
      if (it != free_.end() && it->first <= 16 * std::max(bytes, kSmallest)) {
        void* p = it->second;
        *capacity = it->first;
        kept_ -= it->first;
        free_.erase(it);
        return p;
      }
    }
    size_t cap = kSmallest;
    while (cap < bytes) cap *= 2;
    void* p = nullptr;
    if (cudaHostAlloc(&p, cap, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      throw std::runtime_error("out of pinned host memory (" + std::to_string(cap) + " bytes)");
    }
    *capacity = cap;
    return p;
  }
  void put(void* p, size_t capacity) {
    if (!p) return;
    {
      std::lock_guard<std::mutex> lock(mu_);
      if (kept_ + capacity <= kPinnedKept) {
        free_.emplace(capacity, p);
        kept_ += capacity;
        return;
      }
    }
    cudaFreeHost(p);
  }

 private:
  static constexpr size_t kSmallest = 4096, kPinnedKept = size_t(64) << 20;
  std::mutex mu_;
  std::multimap<size_t, void*> free_;
  size_t kept_ = 0;
};

// Device memory in total: a constant of the device (asking for it takes 20 us)
static size_t total_memory(int dev) {
  static std::mutex mu;
  static std::map<int, size_t> known;
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(dev);
  if (it != known.end()) return it->second;
  size_t fr = 0, total = 0;
  CK(cudaMemGetInfo(&fr, &total));
  known[dev] = total;
  return total;
}

// ------------------------------------------------------------------ backend
class CudaBackend : public Backend {
 public:
  int dev = 0;
  cudaStream_t st = nullptr;
  size_t used = 0;
  std::vector<std::pair<void*, size_t>> live;
  // staging for task lists: a ring of pinned memory and its device copy
  char* dtask = nullptr;
  char* htask = nullptr;
  size_t task_cap = 0, task_pos = 0;
  double* part = nullptr;
  size_t part_cap = 0;
  // profiling
  bool profiling = false;
  struct Rec {
    cudaEvent_t a, b;
    double flops;
    int tag;
  };
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> pool;
  // categories: 0 GEMMs, 1 H_eff psi (with its operand splits), 2 blocking
  // placement, 3 eigensolver (small matrices only), 4 eigensolver
  static constexpr int kTags = 6;
  double acc_ms[kTags] = {0, 0, 0, 0, 0, 0}, acc_flops[kTags] = {0, 0, 0, 0, 0, 0};
  long acc_launch[kTags] = {0, 0, 0, 0, 0, 0};
  cudaEvent_t ev() {
    if (!pool.empty()) {
      cudaEvent_t e = pool.back();
      pool.pop_back();
      return e;
    }
    cudaEvent_t e;
    CK(cudaEventCreate(&e));
    return e;
  }
  void drain() {
    for (auto& r : recs) {
      CK(cudaEventSynchronize(r.b));
      float ms = 0.f;
      CK(cudaEventElapsedTime(&ms, r.a, r.b));
      int t = std::min(kTags - 1, std::max(0, r.tag));
      acc_ms[t] += ms;
      acc_flops[t] += r.flops;
      acc_launch[t] += 1;
      pool.push_back(r.a);
      pool.push_back(r.b);
    }
    recs.clear();
  }
  static constexpr int kSlots = 3;
  cudaEvent_t mb_[kSlots] = {}, me_[kSlots] = {};
  void mark_begin(int slot) override {
    if (slot < 0 || slot >= kSlots) throw std::logic_error("internal: event slot out of range");
    if (!mb_[slot]) {
      CK(cudaEventCreate(&mb_[slot]));
      CK(cudaEventCreate(&me_[slot]));
    }
    CK(cudaEventRecord(mb_[slot], st));
  }
  void mark_stop(int slot) override {
    if (slot < 0 || slot >= kSlots || !mb_[slot]) throw std::logic_error("internal: event slot not started");
    CK(cudaEventRecord(me_[slot], st));
  }
  double mark_ms(int slot) override {
    if (slot < 0 || slot >= kSlots || !mb_[slot]) throw std::logic_error("internal: event slot not started");
    CK(cudaEventSynchronize(me_[slot]));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, mb_[slot], me_[slot]));
    return ms;
  }
  void set_profile(bool on) override {
    drain();
    profiling = on;
    for (int t = 0; t < kTags; ++t) acc_ms[t] = acc_flops[t] = 0, acc_launch[t] = 0;
  }
  void kernel_stats(int t, double* ms, double* flops, long* launches) override {
    drain();
    t = std::min(kTags - 1, std::max(0, t));
    if (ms) *ms = acc_ms[t];
    if (flops) *flops = acc_flops[t];
    if (launches) *launches = acc_launch[t];
  }

  explicit CudaBackend(int device) : dev(device) {
    CK(cudaSetDevice(dev));
    CK(cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking));
    cudaMemPool_t pool;
    CK(cudaDeviceGetDefaultMemPool(&pool, dev));
    uint64_t thr = UINT64_MAX;
    CK(cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &thr));
    total_mem = total_memory(dev);
    CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  }
  int sms = 152;
  int sm_count() const override { return sms; }
  ~CudaBackend() override {
    cudaStreamSynchronize(st);
    if (side) {
      cudaStreamSynchronize(side);
      cudaStreamDestroy(side);
    }
    for (auto& r : recs) { cudaEventDestroy(r.a); cudaEventDestroy(r.b); }
    for (auto e : pool) cudaEventDestroy(e);
    for (int k = 0; k < kSlots; ++k)
      if (mb_[k]) {
        cudaEventDestroy(mb_[k]);
        cudaEventDestroy(me_[k]);
      }
    if (dtask) cudaFreeAsync(dtask, st);
    if (part) cudaFreeAsync(part, st);
    if (dav_dev) cudaFreeAsync(dav_dev, st);
    if (dig_ws) cudaFreeAsync(dig_ws, st);
    if (dflag) cudaFreeAsync(dflag, st);
    cudaStreamSynchronize(st);
    PinnedPool::get().put(htask, task_cap);
    PinnedPool::get().put(dig_err, dig_err_cap);
    PinnedPool::get().put(dav_host, dav_host_cap);
    cudaStreamDestroy(st);
  }
  std::string name() const override { return "cuda"; }
  void* alloc(size_t b) override {
    void* p = try_alloc(b);
    if (!p) {
      if (budget_ && used + b > budget_)
        throw std::runtime_error("out of device memory (budget of " + std::to_string(budget_) + " bytes: " +
                                 std::to_string(used) + " held, " + std::to_string(b) + " requested)");
      throw std::runtime_error("out of device memory (" + std::to_string(b) + " bytes)");
    }
    return p;
  }
  // the same; nullptr when there is no room for it
  void* try_alloc(size_t& b) {
    void* p = nullptr;
    if (b == 0) b = 8;
    while (budget_ && used + b > budget_ && make_room && make_room()) {
    }
    if (budget_ && used + b > budget_) return nullptr;
    if (cudaMallocAsync(&p, b, st) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    count(b);
    live.push_back({p, b});
    return p;
  }
  void count(size_t b) {
    used += b;
    peak_bytes = std::max(peak_bytes, used);
    window_peak = std::max(window_peak, used);
  }
  void free(void* p) override {
    if (!p) return;
    for (size_t i = 0; i < live.size(); ++i)
      if (live[i].first == p) {
        used -= live[i].second;
        live[i] = live.back();
        live.pop_back();
        break;
      }
    CK(cudaFreeAsync(p, st));
  }
  size_t bytes_in_use() const override { return used; }
  // ---- staging to pinned host memory on the side stream
  cudaStream_t side = nullptr;
  cudaStream_t side_stream() {
    if (!side) CK(cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking));
    return side;
  }
  void* stage_out(void* dev, size_t bytes) override {
    if (!dev || bytes == 0) return nullptr;
    cudaStream_t sd = side_stream();
    void* h = nullptr;
    if (cudaMallocHost(&h, bytes) != cudaSuccess) {
      cudaGetLastError();
      throw std::runtime_error("out of pinned host memory (" + std::to_string(bytes) + " bytes)");
    }
    cudaEvent_t e;
    CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    CK(cudaEventRecord(e, st));
    CK(cudaStreamWaitEvent(sd, e, 0));
    CK(cudaEventDestroy(e));
    CK(cudaMemcpyAsync(h, dev, bytes, cudaMemcpyDeviceToHost, sd));
    // the device buffer goes back to the pool after the copy (side-stream order)
    for (size_t i = 0; i < live.size(); ++i)
      if (live[i].first == dev) {
        used -= live[i].second;
        live[i] = live.back();
        live.pop_back();
        break;
      }
    CK(cudaFreeAsync(dev, sd));
    staged_bytes += bytes;
    staged_out_bytes += bytes;
    return h;
  }
  void* stage_in(const void* host, size_t bytes) override {
    if (!host || bytes == 0) return nullptr;
    cudaStream_t sd = side_stream();
    void* d = alloc(bytes);  // main-stream ordered allocation
    cudaEvent_t e;
    CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    CK(cudaEventRecord(e, st));
    CK(cudaStreamWaitEvent(sd, e, 0));
    CK(cudaEventDestroy(e));
    CK(cudaMemcpyAsync(d, host, bytes, cudaMemcpyHostToDevice, sd));
    staged_in_bytes += bytes;
    return d;
  }
  void stage_join() override {
    if (!side) return;
    cudaEvent_t e;
    CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    CK(cudaEventRecord(e, side));
    CK(cudaStreamWaitEvent(st, e, 0));
    CK(cudaEventDestroy(e));
  }
  void host_release(void* host) override {
    if (!host) return;
    if (side) CK(cudaStreamSynchronize(side));
    CK(cudaFreeHost(host));
  }
  size_t total_mem = 0;
  size_t capacity() const override { return total_mem; }
  size_t device_free() const override {
    size_t fr = 0, tot = 0;
    if (cudaMemGetInfo(&fr, &tot) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return fr;
  }
  void memset0(void* p, size_t b) override { if (b) CK(cudaMemsetAsync(p, 0, b, st)); }
  void copy_d2d(void* d, const void* s, size_t b) override {
    if (b) CK(cudaMemcpyAsync(d, s, b, cudaMemcpyDeviceToDevice, st));
  }
  void copy_h2d(void* d, const void* s, size_t b) override {
    if (b) {
      CK(cudaMemcpyAsync(d, s, b, cudaMemcpyHostToDevice, st));
      CK(cudaStreamSynchronize(st));
    }
  }
  void copy_h2d_later(void* d, const void* s, size_t b) override {
    if (b) CK(cudaMemcpyAsync(d, s, b, cudaMemcpyHostToDevice, st));
  }
  void copy_d2h(void* d, const void* s, size_t b) override {
    if (b) {
      CK(cudaMemcpyAsync(d, s, b, cudaMemcpyDeviceToHost, st));
      CK(cudaStreamSynchronize(st));
      check_digits();
    }
  }
  void sync() override { CK(cudaStreamSynchronize(st)); }
  void sync_checked() override {
    CK(cudaStreamSynchronize(st));
    check_digits();
  }
  int* dflag = nullptr;  // device error flag of the bounded waits
  int* flag() {
    if (!dflag) {
      CK(cudaMallocAsync((void**)&dflag, sizeof(int), st));
      CK(cudaMemsetAsync(dflag, 0, sizeof(int), st));
    }
    return dflag;
  }
  void check_device_flag() override {
    if (dig_err) {
      CK(cudaStreamSynchronize(st));
      check_digits();
    }
    if (!dflag) return;
    int h = 0;
    CK(cudaMemcpyAsync(&h, dflag, sizeof(int), cudaMemcpyDeviceToHost, st));
    CK(cudaStreamSynchronize(st));
    if (h != 0) {
      CK(cudaMemsetAsync(dflag, 0, sizeof(int), st));
      throw std::runtime_error("timeout: a bounded wait in the tcgen05 H_eff psi kernel ran out");
    }
  }
  void* stream() override { return (void*)st; }

  // upload a packed task buffer; returns the device base pointer
  char* upload(const std::vector<std::pair<const void*, size_t>>& parts, std::vector<size_t>& offs) {
    size_t tot = 0;
    offs.clear();
    for (auto& p : parts) {
      offs.push_back(tot);
      tot += (p.second + 255) & ~size_t(255);
    }
    if (tot > task_cap) {
      CK(cudaStreamSynchronize(st));
      PinnedPool::get().put(htask, task_cap);
      htask = nullptr;
      const size_t want = std::max(std::max(tot, 2 * task_cap), kTaskRing);
      task_cap = task_pos = 0;
      size_t cap = 0;
      htask = (char*)PinnedPool::get().take(want, &cap);
      if (dtask) CK(cudaFreeAsync(dtask, st));
      dtask = nullptr;
      CK(cudaMallocAsync((void**)&dtask, cap, st));
      task_cap = cap;
    }
    if (task_pos + tot > task_cap) {
      // around the ring: what was uploaded before has been used
      CK(cudaStreamSynchronize(st));
      task_pos = 0;
    }
    char *h = htask + task_pos, *d = dtask + task_pos;
    task_pos += tot;
    for (size_t i = 0; i < parts.size(); ++i) std::memcpy(h + offs[i], parts[i].first, parts[i].second);
    CK(cudaMemcpyAsync(d, h, tot, cudaMemcpyHostToDevice, st));
    return d;
  }
  static constexpr size_t kTaskRing = size_t(4) << 20;  // some hundred lists between two waits

  void place(const std::vector<PlaceGroup>& groups, const std::vector<PlaceSeg>& segs) override {
    std::vector<PlaceTile> tiles;
    for (size_t gi = 0; gi < groups.size(); ++gi) {
      auto& g = groups[gi];
      for (int r = 0; r < g.rows; r += 32)
        for (int c = 0; c < g.cols; c += 32) tiles.push_back({(int)gi, r, c, 0});
      place_bytes += 16.0 * g.rows * g.cols * std::max(1, g.seg_count);
    }
    if (tiles.empty()) return;
    std::vector<size_t> off;
    char* d = upload({{groups.data(), groups.size() * sizeof(PlaceGroup)},
                      {segs.data(), segs.size() * sizeof(PlaceSeg)},
                      {tiles.data(), tiles.size() * sizeof(PlaceTile)}},
                     off);
    Rec* rec = nullptr;
    if (profiling) {
      recs.push_back(Rec{ev(), ev(), 0.0, 2});
      rec = &recs.back();
      CK(cudaEventRecord(rec->a, st));
    }
    place_kernel<<<(unsigned)tiles.size(), 256, 0, st>>>((const PlaceGroup*)(d + off[0]),
                                                          (const PlaceSeg*)(d + off[1]),
                                                          (const PlaceTile*)(d + off[2]));
    if (rec) CK(cudaEventRecord(rec->b, st));
    if (recs.size() > 4096) drain();
    ++launches;
    CK(cudaGetLastError());
  }

  void gemm(const std::vector<GemmGroup>& groups, const std::vector<GemmSeg>& segs,
            Precision prec) override {
    if (groups.empty()) return;
    double fl = 0.0;
    for (auto& g : groups)
      for (int s = g.seg_begin; s < g.seg_begin + g.seg_count; ++s)
        fl += 2.0 * g.m * g.n * segs[s].k;
    gemm_flops += fl;
    if (profiling) {
      // upload first so the events bracket the kernel only
      Rec r{ev(), ev(), fl, tag};
      recs.push_back(r);
      gemm_impl(groups, segs, prec, &recs.back());
      if (recs.size() > 4096) drain();
      return;
    }
    gemm_impl(groups, segs, prec, nullptr);
  }

  // by_entry = false: products of orthogonal matrices (gemm_digits.cuh)
  void gemm_impl(const std::vector<GemmGroup>& groups, const std::vector<GemmSeg>& segs,
                 Precision prec, Rec* rec, bool by_entry = true) {
    if (prec != Precision::FP64) {
      gemm_split_launch(groups, segs, prec, st,
                        [&](const std::vector<std::pair<const void*, size_t>>& parts,
                            std::vector<size_t>& offs) {
                          char* d = upload(parts, offs);
                          if (rec) CK(cudaEventRecord(rec->a, st));
                          return d;
                        });
      ++launches;
      if (rec) CK(cudaEventRecord(rec->b, st));
      return;
    }
    std::vector<char> digits;
    const bool any = choose_digits(groups, segs, digits);
    if (any) {
      if (rec) CK(cudaEventRecord(rec->a, st));
      gemm_digits(groups, segs, digits, by_entry);
    }
    std::vector<GemmTile> tiles;
    for (size_t gi = 0; gi < groups.size(); ++gi) {
      auto& g = groups[gi];
      if (any && digits[gi]) continue;
      for (int r = 0; r < g.m; r += kTM)
        for (int c = 0; c < g.n; c += kTN) tiles.push_back({(int)gi, r, c, 0});
    }
    if (any && tiles.empty()) {
      if (rec) CK(cudaEventRecord(rec->b, st));
      return;
    }
    std::vector<size_t> off;
    char* d = upload({{groups.data(), groups.size() * sizeof(GemmGroup)},
                      {segs.data(), segs.size() * sizeof(GemmSeg)},
                      {tiles.data(), tiles.size() * sizeof(GemmTile)}},
                     off);
    if (rec && !any) CK(cudaEventRecord(rec->a, st));
    // grid.x is limited to 2^31-1; task lists stay far below
    gemm_f64_kernel<<<(unsigned)tiles.size(), 256, 0, st>>>((const GemmGroup*)(d + off[0]),
                                                             (const GemmSeg*)(d + off[1]),
                                                             (const GemmTile*)(d + off[2]));
    ++launches;
    CK(cudaGetLastError());
    if (rec) CK(cudaEventRecord(rec->b, st));
  }

  // Which float64 groups go to the digit products (gemm_digits.cuh): those
  // whose modelled tensor time is below their time on the FMA pipe, if that
  // saves more than the two extra launches of the split (kDigLaunchClocks).
  // The choice depends on the list's shapes only.
  static constexpr double kDigLaunchClocks = 25000.0;
  bool choose_digits(const std::vector<GemmGroup>& groups, const std::vector<GemmSeg>& segs,
                     std::vector<char>& digits) const {
    double df = 0.0, dd = 0.0, tf = 0.0, td = 0.0;
    bool any = false;
    digits.assign(groups.size(), 0);
    for (size_t i = 0; i < groups.size(); ++i) {
      const GemmGroup& g = groups[i];
      if (g.m <= 0 || g.n <= 0 || g.seg_count <= 0) continue;
      const DigCost c = dig_cost(g, segs.data());
      if (c.digits >= c.fma) continue;
      digits[i] = 1;
      any = true;
      df += c.fma;
      dd += c.digits;
      tf = std::max(tf, c.fma_tile);
      td = std::max(td, c.digits_tile / dig_parts(g, segs.data()));
    }
    return any && std::max(dd / sms, td) + kDigLaunchClocks < std::max(df / sms, tf);
  }
  // Digit pool of one launch (bytes): groups are taken until their operands
  // reach it.  It counts against the context's budget like any allocation, and
  // is kept to a sixteenth of it; a single larger group is tried whole, and one
  // that there is no room for runs on the FMA kernel, which needs none.
  size_t dig_pool_cap() const {
    const size_t cap = size_t(2) << 30;
    return budget_ ? std::max<size_t>(size_t(16) << 20, std::min(cap, budget_ / 16)) : cap;
  }
  size_t dig_err_cap = 0;
  int* dig_err = nullptr;  // host-mapped: set by a digit launch whose wait ran out
  void check_digits() {
    if (dig_err && *(volatile int*)dig_err) {
      *dig_err = 0;
      throw std::runtime_error("timeout: a bounded wait in the digit GEMM ran out");
    }
  }
  // clears digits[i] of the groups left to the FMA kernel
  void gemm_digits(const std::vector<GemmGroup>& groups, const std::vector<GemmSeg>& segs,
                   std::vector<char>& digits, bool by_entry) {
    if (!dig_err) {
      dig_err = (int*)PinnedPool::get().take(sizeof(int), &dig_err_cap);
      *dig_err = 0;
    }
    DigPlanner pl;
    const size_t cap = dig_pool_cap();
    std::vector<size_t> planned;
    auto add = [&](size_t i) { pl.add(groups[i], segs.data(), dig_parts(groups[i], segs.data())); };
    auto run = [&]() {
      if (!run_digits(pl.plan, by_entry)) {
        // no room: its groups one by one
        for (size_t i : planned) {
          pl.clear();
          add(i);
          if (planned.size() == 1 || !run_digits(pl.plan, by_entry)) digits[i] = 0;
        }
      }
      pl.clear();
      planned.clear();
    };
    for (size_t i = 0; i < groups.size(); ++i) {
      if (!digits[i]) continue;
      add(i);
      planned.push_back(i);
      if (pl.pool_bytes() >= cap) run();
    }
    run();
  }
  static constexpr size_t kDigKept = size_t(64) << 20;
  char* dig_ws = nullptr;
  size_t dig_ws_cap = 0;
  std::vector<char> dig_zero;
  // false when there is no room for the work space
  bool run_digits(DigPlan& p, bool by_entry) {
    if (p.tasks.empty()) return true;
    // longest tasks first, dealt round-robin over the persistent CTAs
    std::vector<double> w(p.tasks.size());
    std::vector<int> order(p.tasks.size());
    for (size_t t = 0; t < p.tasks.size(); ++t) {
      order[t] = (int)t;
      for (int s = 0; s < p.tasks[t].seg_count; ++s)
        w[t] += std::max(64, p.ops[p.segs[p.tasks[t].seg_begin + s].a].k);
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return w[a] > w[b]; });
    std::vector<DigTask> tasks(p.tasks.size());
    for (size_t t = 0; t < tasks.size(); ++t) tasks[t] = p.tasks[order[t]];
    auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
    const size_t ox = al(p.pool_bytes()), ok = ox + al(p.nexp * sizeof(int));
    const size_t onz = ok + al((p.units + 32) * sizeof(DigMask)), osp = onz + al((p.units + 32) * sizeof(uint16_t));
    const size_t ofl = osp + al((p.ops.size() + 1) * sizeof(int));
    const size_t omi = ofl + al(p.marks), olb = omi + al((size_t)p.marks * 32 * sizeof(uint32_t));
    const size_t osc = olb + al(p.tasks.size() * 8 * sizeof(int));
    // Work space of a launch sequence: small ones share a block that the backend
    // keeps (stream order separates them; not under a budget, which it would
    // take from), larger ones come and go.  The part that starts at zero is
    // uploaded with the lists while it is small.
    char* ws = nullptr;
    size_t bytes = osc + (size_t)p.scratch * sizeof(double);
    const size_t nzero = ofl - osp;
    const bool keep = !budget_ && bytes <= kDigKept;
    if (!keep) {
      ws = (char*)try_alloc(bytes);
      if (!ws) return false;
    } else {
      if (bytes > dig_ws_cap) {
        if (dig_ws) CK(cudaFreeAsync(dig_ws, st));
        dig_ws = nullptr;
        dig_ws_cap = 0;
        const size_t want = std::min(kDigKept, std::max(2 * bytes, size_t(1) << 20));
        if (cudaMallocAsync((void**)&dig_ws, want, st) != cudaSuccess) {
          cudaGetLastError();
          dig_ws = nullptr;
          return false;
        }
        dig_ws_cap = want;
      }
      ws = dig_ws;
      count(bytes);  // what a budget has to leave for this launch
      used -= bytes;
    }
    const bool inline_zero = nzero <= size_t(32) << 10;
    if (inline_zero) dig_zero.resize(std::max(dig_zero.size(), nzero), 0);
    else CK(cudaMemsetAsync(ws + osp, 0, nzero, st));
    std::vector<size_t> off;
    char* d = upload({{p.ops.data(), p.ops.size() * sizeof(DigOperand)},
                      {p.splits.data(), p.splits.size() * sizeof(DigSplit)},
                      {p.segs.data(), p.segs.size() * sizeof(DigSeg)},
                      {tasks.data(), tasks.size() * sizeof(DigTask)},
                      {p.reds.data(), p.reds.size() * sizeof(DigReduce)},
                      {dig_zero.data(), inline_zero ? nzero : 0}},
                     off);
    DigLaunch L{};
    L.ops = (const DigOperand*)(d + off[0]);
    L.splits = (const DigSplit*)(d + off[1]);
    L.segs = (const DigSeg*)(d + off[2]);
    L.tasks = (const DigTask*)(d + off[3]);
    L.reds = (const DigReduce*)(d + off[4]);
    L.nsplits = (int)p.splits.size();
    L.ntasks = (int)tasks.size();
    L.nreds = (int)p.reds.size();
    L.nops = (int)p.ops.size();
    L.pool = (unsigned char*)ws;
    L.last = L.pool + (size_t)p.units * kDigUnit;
    L.exps = (int*)(ws + ox);
    L.masks = (DigMask*)(ws + ok);
    L.nonzero = (uint16_t*)(ws + onz);
    L.by_entry = by_entry;
    L.special = (int*)(inline_zero ? d + off[5] : ws + osp);
    L.flag = (unsigned char*)(ws + ofl);
    L.miss = (uint32_t*)(ws + omi);
    L.left = (int*)(ws + olb);
    L.scratch = (double*)(ws + osc);
    L.err = dig_err;
    L.wait_ns = wait_ns_;
    L.sms = sms;
    dig_launch(L, st);
    launches += 3 + (L.nreds > 0);
    if (!keep) free(ws);
    return true;
  }

  void hpsi(const HpsiBlock* blocks, const HpsiItem* items, const HpsiTask* tasks, int ntasks,
            const HpsiReduce* reds, int nreds, double* scratch, Precision prec, double flops) override {
    gemm_flops += flops;
    Rec* rec = nullptr;
    if (profiling) {
      recs.push_back(Rec{ev(), ev(), flops, 1});
      rec = &recs.back();
      CK(cudaEventRecord(rec->a, st));
    }
    hpsi_launch(blocks, items, tasks, ntasks, reds, nreds, scratch, prec, flag(), st);
    launches += (ntasks > 0) + (nreds > 0);
    if (rec) CK(cudaEventRecord(rec->b, st));
    if (recs.size() > 4096) drain();
  }

  void hpsi_tc(const TcLaunch& L, double flops, int tag) override {
    gemm_flops += flops;
    Rec* rec = nullptr;
    if (profiling) {
      recs.push_back(Rec{ev(), ev(), flops, tag});
      rec = &recs.back();
      CK(cudaEventRecord(rec->a, st));
    }
    hpsi_tc_launch(L, flag(), wait_ns_, st);
    launches += (L.ncta > 0) + (L.nreds > 0);
    if (rec) CK(cudaEventRecord(rec->b, st));
    if (recs.size() > 4096) drain();
  }
  void split(const SplitJob* jobs, int n, float* pool) override {
    if (n <= 0) return;
    // the operand splits of the tcgen05 path (tag 5)
    Rec* rec = nullptr;
    if (profiling) {
      recs.push_back(Rec{ev(), ev(), 0.0, 5});
      rec = &recs.back();
      CK(cudaEventRecord(rec->a, st));
    }
    split_launch(jobs, n, pool, st);
    ++launches;
    if (rec) CK(cudaEventRecord(rec->b, st));
    if (recs.size() > 4096) drain();
  }

  void ensure_part(size_t n) {
    if (n <= part_cap) return;
    if (part) CK(cudaFreeAsync(part, st));
    part_cap = std::max(n, 2 * part_cap);
    CK(cudaMallocAsync((void**)&part, part_cap * sizeof(double), st));
  }
  void dots(const double* V, int m, size_t len, size_t ld, const double* x, double* out) override {
    if (m <= 0) return;
    int nb = (int)std::min<size_t>(kRedBlocks, (len + 255) / 256);
    if (nb < 1) nb = 1;
    ensure_part((size_t)m * nb);
    dots_partial<<<dim3(nb, m), 256, 0, st>>>(V, m, len, ld, x, part);
    ++launches;
    dots_final<<<m, 256, 0, st>>>(part, nb, out);
    ++launches;
    CK(cudaGetLastError());
  }
  void combine(double* y, double beta, const double* V, int m, size_t len, size_t ld,
               const double* c) override {
    int nb = (int)std::min<size_t>(152 * 8, (len + 255) / 256);
    if (nb < 1) nb = 1;
    combine_kernel<<<nb, 256, 0, st>>>(y, beta, V, m, len, ld, c);
    ++launches;
    CK(cudaGetLastError());
  }
  void axpby(double* y, double a, const double* x, double b, size_t len) override {
    int nb = (int)std::min<size_t>(152 * 8, (len + 255) / 256);
    if (nb < 1) nb = 1;
    axpby_kernel<<<nb, 256, 0, st>>>(y, a, x, b, len);
    ++launches;
    CK(cudaGetLastError());
  }
  void precondition(double* y, const double* x, const double* d, double e, size_t len) override {
    int nb = (int)std::min<size_t>(152 * 8, (len + 255) / 256);
    if (nb < 1) nb = 1;
    precond_kernel<<<nb, 256, 0, st>>>(y, x, d, e, len);
    ++launches;
    CK(cudaGetLastError());
  }
  // Davidson: partials, counters and coefficients on the device, results in
  // mapped host memory ([0] |r|^2, [1] the norm, [2 ...] the projections)
  double* dav_dev = nullptr;
  double* dav_host = nullptr;
  size_t dav_host_cap = 0;
  int dav_rows = 0;
  void dav_reserve(int rows) override {
    if (rows <= dav_rows) return;
    CK(cudaStreamSynchronize(st));
    if (dav_dev) CK(cudaFreeAsync(dav_dev, st));
    PinnedPool::get().put(dav_host, dav_host_cap);
    dav_dev = dav_host = nullptr;
    dav_rows = 0;
    rows = std::max(rows, 32);
    // per row: partials, a counter, two coefficients; and |t|^2
    const size_t n = (size_t)rows * (kDavParts + 3) + 1;
    CK(cudaMallocAsync((void**)&dav_dev, n * sizeof(double), st));
    CK(cudaMemsetAsync(dav_dev, 0, n * sizeof(double), st));
    dav_host = (double*)PinnedPool::get().take((size_t)(rows + 2) * sizeof(double), &dav_host_cap);
    dav_rows = rows;
  }
  DavWork dav_work(int m) {
    if (m > dav_rows) throw std::logic_error("internal: Davidson rows beyond the reserved work space");
    return DavWork{dav_dev, (unsigned*)(dav_dev + (size_t)dav_rows * kDavParts), dav_host};
  }
  double* dav_coefs() { return dav_dev + (size_t)dav_rows * (kDavParts + 1); }
  double dav_residual(double* x, double* r, double* t, const double* d, const double* V, const double* HV, int m,
                      size_t len, const double* c, double e) override {
    const DavWork w = dav_work(m);
    if (m > kDavCoefs) {
      CK(cudaMemcpyAsync(dav_coefs(), c, m * sizeof(double), cudaMemcpyHostToDevice, st));
      c = dav_coefs();
    }
    dav_ritz_launch(x, r, t, d, V, HV, m, len, c, e, w, w.host, st);
    ++launches;
    CK(cudaStreamSynchronize(st));
    return ((volatile double*)w.host)[0];
  }
  void dav_orthonormalise(double* V, int m, size_t len, double* in) override {
    const DavWork w = dav_work(m);
    double *t = V + (size_t)m * len, *c = dav_coefs(), *norm2 = c + 2 * (size_t)dav_rows;
    for (int pass = 0; pass < 2; ++pass) {
      dav_dots_launch(V, m, len, t, nullptr, w, c, st);
      dav_subtract_launch(t, V, m, len, c, w, pass ? norm2 : nullptr, st);
    }
    dav_normalise_launch(t, in, len, norm2, w.host + 1, st);
    launches += 5;
  }
  double dav_project(const double* V, int m, size_t len, const double* y, double* hv, double* out) override {
    const DavWork w = dav_work(m);
    dav_dots_launch(V, m, len, y, hv, w, w.host + 2, st);
    ++launches;
    CK(cudaStreamSynchronize(st));
    check_digits();
    for (int i = 0; i < m; ++i) out[i] = ((volatile double*)w.host)[2 + i];
    return ((volatile double*)w.host)[1];
  }
  // Matrices up to kEighSmall (kEighLeaf beside larger ones): one launch of the Jacobi kernel.  Larger ones:
  // cooperative launches of the tridiagonalisation (largest matrices first,
  // group sizes from jac_assign_groups), then the levels of merges with their
  // products on the grouped GEMM, then the reflectors.  Work space (two more
  // copies of the matrices) counts against the budget and is kept to the digit
  // pool's bound, the batch cut into parts of it, and into smaller ones where
  // there is no room; a single matrix runs whole.
  int tri_cap = 0;
  void eigh(const std::vector<EighTask>& tasks) override {
    if (tasks.empty()) return;
    std::vector<EighTask> order(tasks);
    std::stable_sort(order.begin(), order.end(), [](const EighTask& x, const EighTask& y) { return x.n > y.n; });
    while (!order.empty() && order.back().n <= 0) order.pop_back();
    if (order.empty()) return;
    // beside larger matrices the middle ones (17..32) cost nothing there; alone
    // they are faster by Jacobi (one launch)
    const int small = order[0].n > kEighSmall ? kEighLeaf : kEighSmall;
    size_t big = 0;
    while (big < order.size() && order[big].n > small) ++big;
    Rec* rec = nullptr;
    if (profiling) {
      recs.push_back(Rec{ev(), ev(), 0.0, big ? 4 : 3});
      rec = &recs.back();
      CK(cudaEventRecord(rec->a, st));
    }
    if (big < order.size()) {
      std::vector<size_t> off;
      const int count = (int)(order.size() - big);
      char* d = upload({{order.data() + big, count * sizeof(EighTask)}}, off);
      eigh_small_launch((const EighTask*)(d + off[0]), count, st);
      ++launches;
    }
    for (size_t i = 0; i < big;) {
      size_t j = i, bytes = 0;
      for (; j < big; ++j) {
        bytes += 2 * (size_t)order[j].n * order[j].n * sizeof(double);
        if (j > i && bytes > dig_pool_cap()) break;
      }
      eigh_large(std::vector<EighTask>(order.begin() + i, order.begin() + j));
      i = j;
    }
    if (rec) CK(cudaEventRecord(rec->b, st));
    if (recs.size() > 4096) drain();
  }
  void eigh_large(const std::vector<EighTask>& t) {
    if (tri_cap == 0) {
      tri_cap = tridiag_max_ctas(sms);
      if (tri_cap < 2) throw std::runtime_error("cuda: eigensolver needs two co-resident CTAs");
    }
    std::vector<int> sizes;
    size_t sum = 0, sq = 0;
    for (auto& x : t) {
      sizes.push_back(x.n);
      sum += x.n;
      sq += (size_t)x.n * x.n;
    }
    if (sum > (size_t)INT32_MAX) throw std::runtime_error("eigensolver: batch beyond 2^31 rows");
    const DcPlan plan = dc_plan(sizes);
    const std::vector<JacBatch> batches = jac_plan_batches(sizes, tri_cap);
    std::vector<DcNode> nodes = plan.leaves;
    std::vector<size_t> first;
    for (auto& level : plan.merges) {
      first.push_back(nodes.size());
      nodes.insert(nodes.end(), level.begin(), level.end());
    }
    // one allocation: matrices, descriptors, flat arrays
    size_t at = 0;
    auto take = [&](size_t bytes) {
      const size_t o = at;
      at += (bytes + 255) & ~size_t(255);
      return o;
    };
    const size_t oB0 = take(sq * 8), oB1 = take(sq * 8), oP = take(sum * sizeof(unsigned));
    size_t oD[11];
    for (auto& o : oD) o = take(sum * 8);
    const size_t oI = take(3 * sum * 4), oC = take(2 * sum * 4), oR = take(sum * sizeof(DcRot));
    const size_t oW = take(tridiag_wide(sizes[0], (int)sum, tri_cap) * 8);
    const size_t oX = take(8 * sum * 8), obar = take(t.size() * sizeof(unsigned)), osc = take(t.size() * 8);
    const size_t om = take(t.size() * sizeof(DcMatrix)), on = take(nodes.size() * sizeof(DcNode));
    char* ws = t.size() > 1 ? (char*)try_alloc(at) : (char*)alloc(at);
    if (!ws) {
      // no room for all at once
      eigh_large(std::vector<EighTask>(t.begin(), t.begin() + t.size() / 2));
      eigh_large(std::vector<EighTask>(t.begin() + t.size() / 2, t.end()));
      return;
    }
    struct Free {
      CudaBackend* b;
      void* p;
      ~Free() {
        try {
          b->free(p);
        } catch (...) {  // a sticky error is thrown by the next call
        }
      }
    } release{this, ws};
    auto dbl = [&](size_t o) { return (double*)(ws + o); };
    DcArrays ar{};
    ar.d = dbl(oD[0]);
    ar.e = dbl(oD[1]);
    ar.tau = dbl(oD[2]);
    ar.val = dbl(oD[3]);
    ar.dl = dbl(oD[4]);
    ar.zl = dbl(oD[5]);
    ar.mu = dbl(oD[6]);
    ar.zhat = dbl(oD[7]);
    ar.ninv = dbl(oD[8]);
    ar.rho = dbl(oD[9]);
    ar.org = (int*)(ws + oI);
    ar.pos = ar.org + sum;
    ar.inv = ar.pos + sum;
    ar.count = (int*)(ws + oC);
    ar.rot = (DcRot*)(ws + oR);
    ar.scale = dbl(osc);
    ar.wide = dbl(oW);
    std::vector<DcMatrix> mats;
    std::vector<int> ctas;
    size_t sqo = 0;
    int off = 0;
    for (const JacBatch& b : batches) {
      int c = 0;
      for (size_t k = b.begin; k < b.end; ++k) {
        const int n = t[k].n, g = b.g[k - b.begin];
        DcMatrix m{};
        m.A = const_cast<double*>(t[k].A);
        m.w = t[k].w;
        m.V = t[k].V;
        m.B[0] = dbl(oB0) + sqo;
        m.B[1] = dbl(oB1) + sqo;
        m.xch = dbl(oX) + 8 * (size_t)off;
        m.peak = (unsigned*)(ws + oP) + off;
        m.bar = (unsigned*)(ws + obar) + k;
        m.n = n;
        m.off = off;
        m.g = g;
        m.cta0 = c;
        m.rows_in_smem = tridiag_rows_fit(n, g);
        m.levels = dc_levels(n);
        mats.push_back(m);
        c += g;
        off += n;
        sqo += (size_t)n * n;
      }
      ctas.push_back(c);
    }
    std::vector<size_t> uo;
    char* d = upload({{mats.data(), mats.size() * sizeof(DcMatrix)}, {nodes.data(), nodes.size() * sizeof(DcNode)}}, uo);
    CK(cudaMemcpyAsync(ws + om, d + uo[0], mats.size() * sizeof(DcMatrix), cudaMemcpyDeviceToDevice, st));
    CK(cudaMemcpyAsync(ws + on, d + uo[1], nodes.size() * sizeof(DcNode), cudaMemcpyDeviceToDevice, st));
    CK(cudaMemsetAsync(ws + oX, 0, osc - oX, st));  // the exchange and the barriers
    const DcMatrix* dm = (const DcMatrix*)(ws + om);
    const DcNode* dn = (const DcNode*)(ws + on);
    for (size_t b = 0; b < batches.size(); ++b)
      tridiag_launch(dm, (int)batches[b].begin, (int)(batches[b].end - batches[b].begin), ctas[b], ar, flag(),
                     wait_ns_, st);
    dc_leaves_launch(dm, dn, (int)plan.leaves.size(), ar, st);
    launches += (long)batches.size() + 1;
    for (size_t l = 0; l < plan.merges.size(); ++l) {
      const auto& level = plan.merges[l];
      int largest = 0, positions = 0;
      size_t prefix = 0;
      std::vector<GemmGroup> groups;
      std::vector<GemmSeg> segs;
      for (const DcNode& nd : level) {
        const DcMatrix& m = mats[nd.mat];
        const int N = nd.n1 + nd.n2, n = m.n;
        largest = std::max(largest, N);
        positions += N;
        prefix = std::max(prefix, (size_t)(m.B[0] - mats[0].B[0]) + (size_t)n * n);
        const size_t o = (size_t)nd.lo * n + nd.lo, o2 = o + (size_t)nd.n1 * n + nd.n1;
        double* out = m.B[(l + 1) & 1] + o;
        const double* in = m.B[l & 1];
        // rows of the merged vectors: U^T (the children's vectors)
        groups.push_back({out, N, nd.n1, n, (int)segs.size(), 1});
        segs.push_back({m.V + o, in + o, nd.n1, n, n, 1, 0, 1.0});
        groups.push_back({out + nd.n1, N, nd.n2, n, (int)segs.size(), 1});
        segs.push_back({m.V + o + (size_t)nd.n1 * n, in + o2, nd.n2, n, n, 1, 0, 1.0});
      }
      dc_merge_launch(dm, dn + first[l], (int)level.size(), positions, largest, (int)l, ar, st);
      CK(cudaMemsetAsync(mats[0].B[(l + 1) & 1], 0, prefix * sizeof(double), st));
      gemm_impl(groups, segs, Precision::FP64, nullptr, false);
      launches += 6;
    }
    dc_back_launch(dm, (int)mats.size(), (int)sum, sizes[0], ar, st);
    ++launches;
    CK(cudaGetLastError());
  }
};

Backend* make_cuda_backend(int device, std::string* err) {
  int count = 0;
  cudaError_t e = cudaGetDeviceCount(&count);
  if (e != cudaSuccess || count == 0) {
    if (err) *err = std::string("cuda: no usable device (") + cudaGetErrorString(e) + ")";
    cudaGetLastError();
    return nullptr;
  }
  if (device < 0 || device >= count) {
    if (err) *err = "cuda: device ordinal out of range";
    return nullptr;
  }
  try {
    return new CudaBackend(device);
  } catch (const std::exception& ex) {
    if (err) *err = ex.what();
    return nullptr;
  }
}

}  // namespace dmrg
