// Host check of the schedule that a candidate index stands for: the default
// without clusters on blocks of one tile each, with them on blocks of pairs of
// tiles; every other candidate as listed.
#include <cstdio>
#include <vector>

#include "hpsi_tc.cuh"

using namespace dmrg;

int main() {
  int bad = 0;
  static double x;  // an address only
  for (int dim : {40, 512}) {
    std::vector<HpsiBlock> blocks;
    std::vector<HpsiItem> items;
    for (int b = 0; b < 7; ++b) {
      blocks.push_back({&x, dim, dim, dim, (int)items.size(), 5});
      for (int k = 0; k < 5; ++k) items.push_back({&x, &x, &x, dim, dim, dim, 0, 0, dim, dim, 1.0});
    }
    TcPlan plan;
    hpsi_tc_operands(blocks, items, [](size_t) { return (void*)(uintptr_t(1) << 44); }, plan);
    const std::vector<TcShape> c = tc_shape_candidates();
    for (size_t k = 0; k < c.size(); ++k) {
      TcShape want = c[k];
      if (k == 0 && dim == 40) want.cluster = 1;
      const TcShape got = tc_candidate_shape((int)k, blocks, plan.items, [](int cl) { return 152 / cl * cl; });
      if (!(got == want)) {
        std::printf("dim %d candidate %d: cluster %d, not %d\n", dim, (int)k, got.cluster, want.cluster);
        ++bad;
      }
    }
  }
  return bad != 0;
}
