// Host planning of the float64 digit products (gemm_digits.cuh): operands,
// tasks and the cost model that chooses between them and the FMA kernel.
#include <algorithm>

#include "gemm_digits.cuh"

namespace dmrg {

namespace {

// Measured clocks of the kernel: a k-step of a 64-wide tile (bound by shared
// memory: 21 MMAs read 174 KB, the copies write 54 KB), the epilogue of a
// segment behind the next one's k-steps (three float64 operations per output
// at two a clock), and the drain that no k-step overlaps.
constexpr double kStepClocks = 2400.0, kSegClocks = 15000.0, kDrainClocks = 5000.0;
// operands of one group beyond this (bytes of digits) stay on the FMA pipe
constexpr double kMaxPool = 4e9;

// |h| (gemm_digits.cu) gains at most 2^46 a chunk and has to stay below 2^51
constexpr int kDigMaxK = 31 * 256;

}  // namespace

DigCost dig_cost(const GemmGroup& g, const GemmSeg* segs) {
  DigCost c{0, 0, 0, 0};
  double elems = 0.0;
  for (int s = g.seg_begin; s < g.seg_begin + g.seg_count; ++s) {
    const int k = segs[s].k;
    if (k <= 0) continue;
    const double k16 = (k + 15) / 16;
    c.digits_tile += std::max(kStepClocks * k16, kSegClocks) + kDrainClocks;
    c.fma_tile += k16 * 16.0 * 2048.0;
    elems += (double)k * (g.m + g.n);
    if (k > kDigMaxK) c.digits_tile = 1e300;
  }
  if (18.0 * elems > kMaxPool) c.digits_tile = 1e300;
  c.digits = c.digits_tile * ((g.m + kDigTileM - 1) / kDigTileM) * ((g.n + 15) / 16 * 0.25) + 0.6 * elems;
  c.fma = c.fma_tile * ((g.m + 63) / 64) * ((g.n + 63) / 64);
  return c;
}

int dig_parts(const GemmGroup& g, const GemmSeg* segs) {
  (void)segs;
  const int tiles = ((g.m + kDigTileM - 1) / kDigTileM) * ((g.n + kDigTileN - 1) / kDigTileN);
  // a group with few tiles and many segments fills the SMs about twice
  const int want = std::max(1, 304 / std::max(1, tiles));
  return std::max(1, std::min(want, g.seg_count / 2));
}

int DigPlanner::operand(const double* p, int rows, int k, int ld, int trans) {
  const Key key{p, rows, k, ld, trans};
  auto [it, fresh] = seen_.emplace(key, (int)plan.ops.size());
  if (!fresh) return it->second;
  DigOperand o{};
  o.src = p;
  o.rows = rows;
  o.k = k;
  o.ld = ld;
  o.trans = trans;
  o.groups = (rows + 7) / 8;
  o.unit = plan.units;
  o.eoff = plan.nexp;
  o.koff = plan.nkmax;
  plan.units += (long long)((k + 15) / 16) * kDigSums * o.groups;
  plan.nexp += rows;
  plan.nkmax += k;
  for (int r = 0; r < rows; r += 32) plan.splits.push_back({(int)plan.ops.size(), r});
  plan.ops.push_back(o);
  return it->second;
}

void DigPlanner::add(const GemmGroup& g, const GemmSeg* segs, int parts) {
  if (g.m <= 0 || g.n <= 0) return;
  const int first = (int)plan.segs.size();
  for (int s = g.seg_begin; s < g.seg_begin + g.seg_count; ++s) {
    const GemmSeg& x = segs[s];
    if (x.k <= 0) continue;
    // op(A): m x k rows; op(B)^T: n x k rows, stored k x n unless transB
    plan.segs.push_back({operand(x.A, g.m, x.k, x.lda, x.transA), operand(x.B, g.n, x.k, x.ldb, !x.transB), x.alpha});
  }
  const int cnt = (int)plan.segs.size() - first;
  if (cnt == 0) return;
  parts = std::min(parts, cnt);
  const int per = (cnt + parts - 1) / parts;
  parts = (cnt + per - 1) / per;
  for (int r = 0; r < g.m; r += kDigTileM)
    for (int c = 0; c < g.n; c += kDigTileN) {
      if (parts > 1) plan.reds.push_back({g.C, plan.scratch, g.m, g.n, g.ldc, r, c, parts});
      for (int p = 0; p < parts; ++p) {
        const int b = p * per;
        const int segs_here = std::min(per, cnt - b);
        plan.tasks.push_back({g.C, parts > 1 ? plan.scratch : -1, g.m, g.n, g.ldc, r, c, first + b, segs_here,
                              plan.marks});
        plan.marks += 8 * segs_here;
        if (parts > 1) plan.scratch += (long long)kDigTileM * kDigTileN;
      }
    }
}

void DigPlanner::clear() {
  plan = DigPlan();
  seen_.clear();
}

}  // namespace dmrg
