// Host check of small_eigh.hpp: residual, orthogonality, order and sign over
// the sizes of a Davidson subspace and spectra that deflate early or not at
// all.  Backward stable: 30 n eps ||A||.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "small_eigh.hpp"

int main() {
  int bad = 0;
  for (int n = 1; n <= 48; ++n)
    for (int kind = 0; kind < 7; ++kind) {
      std::mt19937 rng(100 * n + kind);
      std::normal_distribution<double> g;
      std::vector<double> a((size_t)n * n, 0.0), w(n), z((size_t)n * n);
      for (int i = 0; i < n; ++i)
        for (int j = 0; j <= i; ++j) {
          double x = 0.0;
          if (kind == 0) x = g(rng);
          if (kind == 1) x = 1.0;
          if (kind == 2) x = i == j ? (double)(rng() % 3) : 0.0;
          if (kind == 3) x = i - j == 1 ? -1.0 : i == j ? 2.0 : 0.0;
          if (kind == 4) x = g(rng) * std::pow(10.0, -(i + j) / 3.0);
          // the subspace matrix of a converging iteration: weak last row
          if (kind == 5) x = i == j ? -50.0 + 2.0 * i : i == n - 1 ? 1e-9 * g(rng) : 1e-14 * g(rng);
          if (kind == 6) x = 1e-200 * g(rng);
          a[(size_t)i * n + j] = a[(size_t)j * n + i] = x;
        }
      dmrg::small_eigh(n, a.data(), w.data(), z.data());
      double norm = 1e-300;
      for (double x : w) norm = std::max(norm, std::abs(x));
      const double tol = 30.0 * n * 2.2e-16;
      for (int r = 0; r < n; ++r) {
        if (r && w[r] < w[r - 1]) ++bad;
        double top = 0.0, sign = 1.0;
        for (int i = 0; i < n; ++i) {
          double y = 0.0, o = 0.0;
          for (int j = 0; j < n; ++j) {
            y += a[(size_t)i * n + j] * z[(size_t)r * n + j];
            o += z[(size_t)i * n + j] * z[(size_t)r * n + j];
          }
          const double x = z[(size_t)r * n + i];
          if (std::abs(x) > top + 1e-12) top = std::abs(x), sign = x;
          if (!(std::abs(y - w[r] * x) <= tol * norm) || !(std::abs(o - (i == r)) <= tol)) ++bad;
        }
        if (sign <= 0.0) ++bad;
      }
    }
  // meaningless input ends
  std::vector<double> a(25, NAN), w(5), z(25);
  dmrg::small_eigh(5, a.data(), w.data(), z.data());
  if (bad) {
    std::printf("%d failures\n", bad);
    return 1;
  }
  std::printf("small eigensolver checks passed\n");
  return 0;
}
