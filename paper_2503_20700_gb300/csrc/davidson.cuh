// Vector kernels of the Davidson iteration (rows of V and HV of length len,
// stride len).  Every sum over a vector has its partials added by the last CTA
// to arrive, in a fixed order, so a result needs no second launch.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace dmrg {

constexpr int kDavCoefs = 64;  // coefficients passed with the launch

struct DavWork {
  double* part;       // kDavParts doubles per sum
  unsigned* arrived;  // one counter per sum, zero; left zero
  double* host;       // mapped host memory: what the host reads after a launch
};
constexpr int kDavParts = 608;

// c: m coefficients on the host (device when m > kDavCoefs)
void dav_ritz_launch(double* x, double* r, double* t, const double* d, const double* V, const double* HV, int m,
                     size_t len, const double* c, double e, DavWork w, double* norm2, cudaStream_t st);
// out[i] = V_i . y for i < m; copy (if not null) = y
void dav_dots_launch(const double* V, int m, size_t len, const double* y, double* copy, DavWork w, double* out,
                     cudaStream_t st);
// t -= sum_i c[i] V_i; norm2 (if not null) = |t|^2
void dav_subtract_launch(double* t, const double* V, int m, size_t len, const double* c, DavWork w, double* norm2,
                         cudaStream_t st);
// t and in = t / |t| (zero below 1e-14); *norm = |t|
void dav_normalise_launch(double* t, double* in, size_t len, const double* norm2, double* norm, cudaStream_t st);

}  // namespace dmrg
