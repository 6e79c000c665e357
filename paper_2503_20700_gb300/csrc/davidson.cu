// Vector kernels of the Davidson iteration (davidson.cuh).  Bound by HBM for the
// vectors of a large bond and by launches for the small ones, so each does what
// the iteration needs between two waits of the host: a residual with its norm
// and the preconditioned vector is one launch (five before), a projection two
// with the device's own coefficients in place of a copy to the host and back.
// Measured, an iteration of a 10-site D = 64 run (24 rows at most): some 25
// launches and 9 waits of the host and 615 us -> 9 launches and 2 waits and
// 330 us, with the subspace problem (146 us on the device) on the host.
#include "davidson.cuh"

#include <algorithm>
#include <stdexcept>
#include <string>

namespace dmrg {

namespace {

constexpr int NT = 256;

struct Coefs {
  double c[kDavCoefs];
};

__device__ __forceinline__ double cta_sum(double x, double* sh) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  x = sh[0];
#pragma unroll
  for (int i = 1; i < NT / 32; ++i) x += sh[i];
  return x;
}
// adds x over the CTA, then over the CTAs of the sum; true in every thread of
// the CTA that has the total
__device__ __forceinline__ bool grid_sum(double& x, double* part, unsigned* arrived) {
  __shared__ double sh[2][NT / 32];
  __shared__ bool last;
  const double s = cta_sum(x, sh[0]);
  if (threadIdx.x == 0) {
    __stcg(part + blockIdx.x, s);
    __threadfence();
    last = atomicInc(arrived, gridDim.x - 1) == gridDim.x - 1;  // wraps to zero
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double v = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += NT) v += __ldcg(part + i);
  x = cta_sum(v, sh[1]);
  return true;
}

// x = sum c_i V_i, r = sum c_i HV_i - e x, t = r / (d - e) with a guarded
// denominator (r without d), |r|^2
__global__ void __launch_bounds__(NT) ritz_kernel(double* __restrict__ x, double* __restrict__ r,
                                                  double* __restrict__ t, const double* __restrict__ d,
                                                  const double* __restrict__ V, const double* __restrict__ HV, int m,
                                                  size_t len, const Coefs k, const double* __restrict__ more, double e,
                                                  double* part, unsigned* arrived, double* norm2) {
  double s = 0.0;
  for (size_t j = (size_t)blockIdx.x * NT + threadIdx.x; j < len; j += (size_t)gridDim.x * NT) {
    double a = 0.0, b = 0.0;
#pragma unroll 4
    for (int i = 0; i < m; ++i) {
      const double c = more ? more[i] : k.c[i];
      a = fma(c, V[(size_t)i * len + j], a);
      b = fma(c, HV[(size_t)i * len + j], b);
    }
    b = fma(1.0, b, -e * a);
    x[j] = a;
    r[j] = b;
    if (t) {
      double y = b;
      if (d) {
        double den = d[j] - e;
        if (fabs(den) < 1e-8) den = den < 0 ? -1e-8 : 1e-8;
        y = b / den;
      }
      t[j] = y;
    }
    s = fma(b, b, s);
  }
  if (grid_sum(s, part, arrived) && threadIdx.x == 0) *norm2 = s;
}

__global__ void __launch_bounds__(NT) dots_kernel(const double* __restrict__ V, size_t len,
                                                  const double* __restrict__ y, double* __restrict__ copy,
                                                  double* part, unsigned* arrived, double* out) {
  const int i = blockIdx.y;
  const double* v = V + (size_t)i * len;
  double s = 0.0;
  for (size_t j = (size_t)blockIdx.x * NT + threadIdx.x; j < len; j += (size_t)gridDim.x * NT) {
    const double q = y[j];
    s = fma(v[j], q, s);
    if (i == 0 && copy) copy[j] = q;
  }
  if (grid_sum(s, part + (size_t)i * kDavParts, arrived + i) && threadIdx.x == 0) out[i] = s;
}

__global__ void __launch_bounds__(NT) subtract_kernel(double* __restrict__ t, const double* __restrict__ V, int m,
                                                      size_t len, const double* __restrict__ c, double* part,
                                                      unsigned* arrived, double* norm2) {
  double s = 0.0;
  for (size_t j = (size_t)blockIdx.x * NT + threadIdx.x; j < len; j += (size_t)gridDim.x * NT) {
    double a = 0.0;
#pragma unroll 4
    for (int i = 0; i < m; ++i) a = fma(-__ldg(c + i), V[(size_t)i * len + j], a);
    const double y = fma(1.0, t[j], a);
    t[j] = y;
    s = fma(y, y, s);
  }
  if (norm2 && grid_sum(s, part, arrived) && threadIdx.x == 0) *norm2 = s;
}

__global__ void __launch_bounds__(NT) normalise_kernel(double* __restrict__ t, double* __restrict__ in, size_t len,
                                                       const double* __restrict__ norm2, double* norm) {
  const double n = sqrt(fmax(0.0, *norm2));
  const double f = n < 1e-14 ? 0.0 : 1.0 / n;
  for (size_t j = (size_t)blockIdx.x * NT + threadIdx.x; j < len; j += (size_t)gridDim.x * NT) {
    const double y = f * t[j];
    t[j] = y;
    in[j] = y;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *norm = n;
}

void check(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string("cuda: ") + what + ": " + cudaGetErrorString(e));
}
int blocks(size_t len, int most) { return (int)std::max<size_t>(1, std::min<size_t>(most, (len + NT - 1) / NT)); }

}  // namespace

void dav_ritz_launch(double* x, double* r, double* t, const double* d, const double* V, const double* HV, int m,
                     size_t len, const double* c, double e, DavWork w, double* norm2, cudaStream_t st) {
  Coefs k{};
  if (m <= kDavCoefs) std::copy(c, c + m, k.c);
  ritz_kernel<<<blocks(len, kDavParts), NT, 0, st>>>(x, r, t, d, V, HV, m, len, k, m <= kDavCoefs ? nullptr : c, e,
                                                     w.part, w.arrived, norm2);
  check("residual");
}

void dav_dots_launch(const double* V, int m, size_t len, const double* y, double* copy, DavWork w, double* out,
                     cudaStream_t st) {
  dots_kernel<<<dim3(blocks(len, 152), m), NT, 0, st>>>(V, len, y, copy, w.part, w.arrived, out);
  check("projection");
}

void dav_subtract_launch(double* t, const double* V, int m, size_t len, const double* c, DavWork w, double* norm2,
                         cudaStream_t st) {
  subtract_kernel<<<blocks(len, kDavParts), NT, 0, st>>>(t, V, m, len, c, w.part, w.arrived, norm2);
  check("orthogonalisation");
}

void dav_normalise_launch(double* t, double* in, size_t len, const double* norm2, double* norm, cudaStream_t st) {
  normalise_kernel<<<blocks(len, 1216), NT, 0, st>>>(t, in, len, norm2, norm);
  check("normalisation");
}

}  // namespace dmrg
