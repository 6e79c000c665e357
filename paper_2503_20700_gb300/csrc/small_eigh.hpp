// Symmetric eigenproblem of a Davidson subspace on the host (at most some tens
// of rows): Householder tridiagonalisation and the implicit QR step with
// Wilkinson's shift (Golub and Van Loan, Matrix Computations, 8.3).
//
// On the host because it is one serial chain: a square root or a division of
// a rotation takes the GPU's float64 pipe hundreds of clocks, and every output
// (coefficients, energy, convergence) is needed on the host anyway.
#pragma once
#include <algorithm>
#include <cmath>
#include <limits>
#include <numeric>
#include <vector>

namespace dmrg {

// w: eigenvalues ascending; z: eigenvectors as rows, the component of largest
// magnitude positive.  a: n x n row-major, symmetric.
inline void small_eigh(int n, const double* a, double* w, double* z) {
  std::vector<double> t(a, a + (size_t)n * n), d(n), e(n, 0.0), q((size_t)n * n, 0.0), p(n);
  std::vector<double> tau(n, 0.0);
  // divided by a power of two that brings the largest entry to about one
  double top = 0.0;
  for (double x : t) top = std::max(top, std::abs(x));
  const int ex = top > 0.0 && std::isfinite(top) ? std::ilogb(top) : 0;
  for (double& x : t) x = std::ldexp(x, -ex);
  // column k below the diagonal keeps reflector k in row k of t
  for (int k = 0; k + 2 < n; ++k) {
    double* v = &t[(size_t)k * n];
    double s = 0.0;
    for (int j = k + 2; j < n; ++j) s += v[j] * v[j];
    e[k] = v[k + 1];
    // a tail below 1e-30 of the matrix is left out (its squares would lose
    // digits to underflow)
    if (!(s > 1e-60)) continue;
    const double beta = -std::copysign(std::sqrt(v[k + 1] * v[k + 1] + s), v[k + 1]);
    tau[k] = (beta - v[k + 1]) / beta;
    const double f = 1.0 / (v[k + 1] - beta);
    for (int j = k + 2; j < n; ++j) v[j] *= f;
    v[k + 1] = 1.0;
    e[k] = beta;
    double pv = 0.0;
    for (int i = k + 1; i < n; ++i) {
      double y = 0.0;
      for (int j = k + 1; j < n; ++j) y += t[(size_t)i * n + j] * v[j];
      p[i] = tau[k] * y;
      pv += p[i] * v[i];
    }
    const double h = 0.5 * tau[k] * pv;
    for (int i = k + 1; i < n; ++i) p[i] -= h * v[i];
    for (int i = k + 1; i < n; ++i)
      for (int j = k + 1; j < n; ++j) t[(size_t)i * n + j] -= v[i] * p[j] + p[i] * v[j];
  }
  if (n >= 2) e[n - 2] = t[(size_t)(n - 2) * n + n - 1];
  for (int i = 0; i < n; ++i) {
    d[i] = t[(size_t)i * n + i];
    q[(size_t)i * n + i] = 1.0;
  }
  // rows of q: columns of the product of the reflectors
  for (int k = n - 3; k >= 0; --k) {
    if (tau[k] == 0.0) continue;
    const double* v = &t[(size_t)k * n];
    for (int r = k + 1; r < n; ++r) {
      double* x = &q[(size_t)r * n];
      double s = 0.0;
      for (int j = k + 1; j < n; ++j) s += x[j] * v[j];
      s *= tau[k];
      for (int j = k + 1; j < n; ++j) x[j] -= s * v[j];
    }
  }
  const double eps = std::numeric_limits<double>::epsilon();
  int hi = n - 1;
  for (int step = 0; hi > 0 && step < 60 * n; ++step) {
    auto negligible = [&](int k) { return std::abs(e[k]) <= eps * (std::abs(d[k]) + std::abs(d[k + 1])); };
    if (negligible(hi - 1)) {
      --hi;
      continue;
    }
    int lo = hi - 1;
    while (lo > 0 && !negligible(lo - 1)) --lo;
    // the eigenvalue of the last 2 x 2 block nearer to its last entry
    const double b = e[hi - 1], g = 0.5 * (d[hi - 1] - d[hi]);
    const double shift = d[hi] - b * b / (g + std::copysign(std::hypot(g, b), g));
    double x = d[lo] - shift, y = e[lo];
    for (int k = lo; k < hi; ++k) {
      const double r = std::hypot(x, y), c = r > 0.0 ? x / r : 1.0, s = r > 0.0 ? y / r : 0.0;
      if (k > lo) e[k - 1] = r;
      const double dk = d[k], dn = d[k + 1], ek = e[k], m = 2.0 * c * s * ek;
      d[k] = c * c * dk + m + s * s * dn;
      d[k + 1] = s * s * dk - m + c * c * dn;
      e[k] = c * s * (dn - dk) + (c * c - s * s) * ek;
      if (k + 1 < hi) {
        x = e[k];
        y = s * e[k + 1];
        e[k + 1] *= c;
      }
      double *u = &q[(size_t)k * n], *v = u + n;
      for (int j = 0; j < n; ++j) {
        const double uj = u[j], vj = v[j];
        u[j] = c * uj + s * vj;
        v[j] = c * vj - s * uj;
      }
    }
  }
  std::vector<int> order(n);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int i, int j) { return d[i] < d[j]; });
  for (int r = 0; r < n; ++r) {
    const double* x = &q[(size_t)order[r] * n];
    int big = 0;
    for (int j = 1; j < n; ++j)
      if (std::abs(x[j]) > std::abs(x[big]) + 1e-12) big = j;
    const double sg = x[big] < 0.0 ? -1.0 : 1.0;
    w[r] = std::ldexp(d[order[r]], ex);
    for (int j = 0; j < n; ++j) z[(size_t)r * n + j] = sg * x[j];
  }
}

}  // namespace dmrg
