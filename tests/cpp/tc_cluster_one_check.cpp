// Host check of schedules without clusters and of the rule that picks them
// (tc_sized_shape): plans of clusters of one pass tc_plan_check and have the
// tasks and partial tiles of the clustered plan; single-tile blocks leave the
// clusters, wide ones keep them.
#include <cstdio>
#include <random>
#include <vector>

#include "hpsi_tc.cuh"

using namespace dmrg;

static int bad = 0;
#define CHECK(x) \
  do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++bad; } } while (0)

static void make(std::mt19937& rng, int lo, int hi, int count, std::vector<HpsiBlock>& blocks,
                 std::vector<HpsiItem>& items) {
  static double a, p, b, c;  // addresses only
  for (int i = 0; i < count; ++i) {
    HpsiBlock bk{&c, lo + (int)(rng() % (hi - lo + 1)), lo + (int)(rng() % (hi - lo + 1)), 0, (int)items.size(),
                 1 + (int)(rng() % 30)};
    bk.ldc = bk.n;
    for (int k = 0; k < bk.item_count; ++k) {
      const int ka = lo + (int)(rng() % (hi - lo + 1)), kb = lo + (int)(rng() % (hi - lo + 1));
      items.push_back({&a, &p, &b, ka, kb, kb, 0, 0, ka, kb, 1.0});
    }
    blocks.push_back(bk);
  }
}

int main() {
  for (unsigned seed = 1; seed <= 20; ++seed)
    for (int hi : {8, 90, 128, 300, 700}) {
      std::mt19937 rng(seed);
      std::vector<HpsiBlock> blocks;
      std::vector<HpsiItem> items;
      make(rng, std::max(1, hi / 4), hi, 1 + (int)(rng() % 12), blocks, items);
      TcPlan one, two;
      void* pool = (void*)(uintptr_t(1) << 44);
      hpsi_tc_operands(blocks, items, [&](size_t) { return pool; }, one);
      hpsi_tc_operands(blocks, items, [&](size_t) { return pool; }, two);
      TcShape s1, s2;
      s1.cluster = 1;
      hpsi_tc_schedule(blocks, one, s1, 152);
      hpsi_tc_schedule(blocks, two, s2, 152);
      CHECK(tc_plan_check(one, blocks).empty());
      CHECK(one.scratch == two.scratch && one.tasks.size() == two.tasks.size());
      for (size_t t = 0; t < one.tasks.size() && t < two.tasks.size(); ++t)
        CHECK(one.tasks[t].it_begin == two.tasks[t].it_begin && one.tasks[t].it_count == two.tasks[t].it_count &&
              one.tasks[t].part == two.tasks[t].part);
      for (const TcSlot& s : one.cta_task) CHECK(!s.ghost && s.grpn == 1);
      const TcShape r = tc_sized_shape(s2, blocks, two.items, 152, 152);
      if (hi <= 128) CHECK(r.cluster == 1);
      TcShape four = s2;
      four.cluster = 4;
      CHECK(tc_sized_shape(four, blocks, two.items, 152, 152) == four);
    }
  // pairs of column tiles: clusters stay
  std::vector<HpsiBlock> blocks;
  std::vector<HpsiItem> items;
  std::mt19937 rng(3);
  make(rng, 480, 512, 6, blocks, items);
  TcPlan plan;
  hpsi_tc_operands(blocks, items, [&](size_t) { return (void*)(uintptr_t(1) << 44); }, plan);
  CHECK(tc_sized_shape(TcShape(), blocks, plan.items, 152, 152) == TcShape());
  if (!bad) std::printf("cluster checks passed\n");
  return bad != 0;
}
