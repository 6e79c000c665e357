// Checks of the digit GEMM planner on the CPU (no device calls), over random
// lists of groups with shared operands: the units of the operands are
// disjoint runs of 8 ceil(rows/8) ceil(k/16) that fill the pool; exponents and
// column maxima are disjoint ranges; every operand's rows are split once; the
// tasks of a group cover each 128 x 64 tile and each of its segments once, in
// order, with a partial tile each (and one reduction per tile) when a tile has
// several; a group's segments and parts do not depend on what was planned
// before it.
#include <cstdio>
#include <map>
#include <random>
#include <set>
#include <tuple>
#include <vector>

#include "gemm_digits.cuh"

using namespace dmrg;

static int fails = 0;
#define CHECK(c)                                                \
  do {                                                          \
    if (!(c)) {                                                 \
      std::printf("FAIL %s:%d %s\n", __FILE__, __LINE__, #c);  \
      ++fails;                                                  \
    }                                                           \
  } while (0)

int main() {
  std::mt19937 rng(11);
  auto uni = [&](int a, int b) { return a + (int)(rng() % (unsigned)(b - a + 1)); };
  std::vector<double> mem(1 << 20), out(1 << 20);
  for (int rep = 0; rep < 200; ++rep) {
    std::vector<GemmGroup> gs;
    std::vector<GemmSeg> segs;
    const int ng = uni(1, 12);
    for (int g = 0; g < ng; ++g) {
      const int m = uni(1, 300), n = uni(1, 200), ns = uni(0, rep % 3 ? 3 : 40);
      gs.push_back({out.data() + 1000 * g, m, n, n, (int)segs.size(), ns});
      for (int s = 0; s < ns; ++s) {
        const int k = uni(0, 20) ? uni(1, 500) : 0, ta = uni(0, 1), tb = uni(0, 1);
        segs.push_back({mem.data() + uni(0, 5), mem.data() + uni(0, 5), k, ta ? m : std::max(k, 1),
                        tb ? std::max(k, 1) : n, ta, tb, 0.5});
      }
    }
    DigPlanner all;
    for (auto& g : gs) {
      const size_t t0 = all.plan.tasks.size(), r0 = all.plan.reds.size();
      const int parts = dig_parts(g, segs.data());
      all.add(g, segs.data(), parts);
      DigPlanner one;
      one.add(g, segs.data(), parts);
      CHECK(all.plan.tasks.size() - t0 == one.plan.tasks.size());
      CHECK(all.plan.reds.size() - r0 == one.plan.reds.size());
      std::vector<const GemmSeg*> live;
      for (int s = 0; s < g.seg_count; ++s)
        if (segs[g.seg_begin + s].k > 0) live.push_back(&segs[g.seg_begin + s]);
      std::map<std::pair<int, int>, int> next;  // segments covered so far, by tile
      for (size_t t = t0; t < all.plan.tasks.size(); ++t) {
        const DigTask &a = all.plan.tasks[t], &b = one.plan.tasks[t - t0];
        CHECK(a.seg_count == b.seg_count && a.r0 == b.r0 && a.c0 == b.c0 && (a.part < 0) == (b.part < 0));
        CHECK(a.seg_count > 0 && a.r0 % kDigTileM == 0 && a.c0 % kDigTileN == 0 && a.r0 < g.m && a.c0 < g.n);
        CHECK(a.C == g.C && a.m == g.m && a.n == g.n && a.ldc == g.ldc);
        int& done = next[{a.r0, a.c0}];
        for (int s = 0; s < a.seg_count; ++s, ++done) {
          const DigSeg& d = all.plan.segs[a.seg_begin + s];
          const GemmSeg& x = *live[done];
          const DigOperand &oa = all.plan.ops[d.a], &ob = all.plan.ops[d.b];
          CHECK(oa.src == x.A && oa.rows == g.m && oa.k == x.k && oa.ld == x.lda && oa.trans == x.transA);
          CHECK(ob.src == x.B && ob.rows == g.n && ob.k == x.k && ob.ld == x.ldb && ob.trans == !x.transB);
          CHECK(d.alpha == x.alpha);
        }
      }
      const size_t tiles = live.empty() ? 0 : (size_t)((g.m + 127) / 128) * ((g.n + 63) / 64);
      CHECK(next.size() == tiles);
      for (auto& kv : next) CHECK(kv.second == (int)live.size());
    }
    const DigPlan& p = all.plan;
    long long unit = 0;
    int e = 0, k = 0;
    std::map<int, std::set<int>> rows;
    for (auto& s : p.splits) CHECK(s.r0 % 32 == 0 && rows[s.op].insert(s.r0).second);
    for (size_t i = 0; i < p.ops.size(); ++i) {
      const DigOperand& o = p.ops[i];
      CHECK(o.unit == unit && o.eoff == e && o.koff == k && o.groups == (o.rows + 7) / 8);
      unit += 8LL * o.groups * ((o.k + 15) / 16);
      e += o.rows;
      k += o.k;
      CHECK((int)rows[(int)i].size() == (o.rows + 31) / 32);
    }
    CHECK(unit == p.units && e == p.nexp && k == p.nkmax);
    std::set<long long> parts;
    std::map<std::tuple<double*, int, int>, std::vector<long long>> by;
    for (auto& t : p.tasks)
      if (t.part >= 0) {
        CHECK(t.part % (kDigTileM * kDigTileN) == 0 && t.part + kDigTileM * kDigTileN <= p.scratch);
        CHECK(parts.insert(t.part).second);
        by[{t.C, t.r0, t.c0}].push_back(t.part);
      }
    CHECK((long long)parts.size() * kDigTileM * kDigTileN == p.scratch && by.size() == p.reds.size());
    for (auto& r : p.reds) {
      const auto& v = by[{r.C, r.r0, r.c0}];
      CHECK((int)v.size() == r.nparts && r.nparts > 1);
      for (size_t i = 0; i < v.size(); ++i) CHECK(v[i] == r.part0 + (long long)i * kDigTileM * kDigTileN);
    }
  }
  std::printf(fails ? "%d failures\n" : "digit plan checks passed\n", fails);
  return fails != 0;
}
