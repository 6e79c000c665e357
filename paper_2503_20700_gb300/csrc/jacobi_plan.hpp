// Host planning of the batched tridiagonalisation (the density-matrix sectors
// of a decimation): which matrices share a cooperative launch of one CTA per
// SM, and how many CTAs each matrix gets.  (The names are those of the solver by
// rotations that it planned for first.)
#pragma once
#include <algorithm>
#include <stdexcept>
#include <vector>

namespace dmrg {

constexpr int kJacSmemN = 112;  // largest matrix that may stay on one CTA

// Modelled time of an n x n matrix on g CTAs, in SM clocks: n steps of three
// float64 FMAs per entry of the trailing matrix (n^2 / 3 entries on average,
// two FMAs a clock), what every CTA repeats (about 4500 clocks) and, in a
// group, the exchange (about 4000: the trip of a published value through L2 and
// the waits around it); the group sizes of a batch minimise the slowest matrix.
inline double jac_cost(int n, int g) {
  const double steps = std::max(1, n - 1);
  const double fma = 0.5 * (double)n * n;
  return steps * (g == 1 ? fma + 4500.0 : fma / g + 8500.0);
}

// g[k] of batch tasks (descending n) start at their minimum; spare CTAs go to
// the slowest matrix while that shortens it
inline void jac_assign_groups(const std::vector<int>& n, std::vector<int>& g, int spare) {
  while (spare > 0 && !n.empty()) {
    size_t k = 0;
    for (size_t i = 1; i < n.size(); ++i)
      if (jac_cost(n[i], g[i]) > jac_cost(n[k], g[k])) k = i;
    const int gmax = std::max(2, std::min(std::max(32, n[k] / 16), ((n[k] + 1) & ~1) / 2));
    int ng = g[k] + 1;
    while (ng <= gmax && ng - g[k] <= spare && jac_cost(n[k], ng) >= jac_cost(n[k], g[k])) ++ng;
    if (ng > gmax || ng - g[k] > spare) break;
    spare -= ng - g[k];
    g[k] = ng;
  }
}

// One cooperative launch: matrices [begin, end) of the size-sorted list and
// the CTA group size of each.
struct JacBatch {
  size_t begin = 0, end = 0;
  std::vector<int> g;
};

// Splits matrices sorted by decreasing n into launches of at most `cap`
// co-resident CTAs (a matrix above kJacSmemN needs a group of at least two)
// and sizes the groups of each launch.
inline std::vector<JacBatch> jac_plan_batches(const std::vector<int>& n_desc, int cap) {
  std::vector<JacBatch> out;
  size_t i0 = 0;
  while (i0 < n_desc.size()) {
    JacBatch b;
    b.begin = i0;
    std::vector<int> ns;
    int used = 0;
    size_t i1 = i0;
    while (i1 < n_desc.size()) {
      const int gmin = n_desc[i1] > kJacSmemN ? 2 : 1;
      if (used + gmin > cap) break;
      ns.push_back(n_desc[i1]);
      b.g.push_back(gmin);
      used += gmin;
      ++i1;
    }
    if (i1 == i0) throw std::runtime_error("eigensolver: fewer co-resident CTAs than one matrix needs");
    jac_assign_groups(ns, b.g, cap - used);
    b.end = i1;
    out.push_back(std::move(b));
    i0 = i1;
  }
  return out;
}

}  // namespace dmrg
