// Float64 grouped GEMM on the bf16 tensor cores by exact digit products (the
// error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59
// (2012) 95, with one exponent per operand row and balanced base-256 digits).
//
//   C += sum_s alpha_s op_s(A_s) op_s(B_s)
//
// Row i of op(A) (column j of op(B)) has one exponent e with |x| < 2^e; every
// entry becomes the integer F = round(x 2^(70-e)), cut into nine balanced
// digits of eight bits, which are stored with their weights 2^-8i (bf16 holds
// them exactly).  The 45 products of digits i and j with i + j = d <= 8 are
// summed by tcgen05.mma into FP32 accumulators: one per d up to 6, and one for 7
// and 8 together (eight are all of TMEM).  256 terms of an accumulator stay below
// 2^24.6 of its unit, below 2^24 for d <= 3, so the sums up to d = 6 are exact
// (a worst case of aligned digits may round in the last place above d = 3, at
// 2^-52 of the row maxima's product and less); the last one carries d = 8 in the
// bits that it has below its unit, 2^-68 of that product, and is rounded to it.
// The accumulators are combined in integers, and each segment is added to the
// output tile in float64.
//
// Precision.  Per term, what the digits drop is of the size of 2^-69 of the
// product of the two rows' maxima 2^ea 2^eb (at most 2^-66), whatever the term
// itself: far below the rounding of a float64 FMA chain where the row maxima
// meet entries of their size, and more than the term where they do not.  So an
// output is taken from the digits only if some term of it is at least 2^-14 of
// 2^ea 2^eb (DigMask), or all its terms are zero.  What is off is then at most
// 2 k 2^-53 of sum |a b|, and measured it is smaller than the error of an FMA
// chain, in the corner of that rule too (a dominant term of 2^-14 and 16 to 200
// in all: 0.1 to 0.4 of the chain's; normal numbers: 0.2).  The other outputs,
// and those of a segment with a non-finite entry or a row maximum outside
// 2^+-400, are left out and marked, and a second kernel adds them by float64
// FMAs (fma_missing_kernel).  A caller whose results are only as good as the norm of
// the rows anyway (products of orthogonal matrices) may have all outputs from
// the digits (by_entry = false).
//
// Nine digits rather than eight (36 products, rule at 2^-7): a k-step takes a
// fifth longer, but rotations near the identity and matrices that decay from
// their diagonal, many of whose outputs eight digits hold less well than FMAs,
// need the FMA pipe no more.  Measured, the rotation of 600 Cholesky vectors of
// 200 orbitals by exp(-K), K = 0.01 N(0, 1): 16.4 ms with eight digits and that
// rule, 1.8 ms with nine (26 ms by FMAs alone); its errors in units of
// 2^-53 sum |a b| 0.11 (root mean square) against 1.09 by FMAs.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <unordered_map>
#include <vector>

#include "backend.hpp"

namespace dmrg {

constexpr int kDigTileM = 128, kDigTileN = 64;  // output tile of a task
constexpr int kDigSlices = 9;
constexpr int kDigSums = kDigSlices - 1;  // accumulators; digits laid out together
constexpr int kDigUnit = 256;  // bytes: 8 rows x 16 columns of one digit

// One operand: rows x k, element (r, c) = trans ? src[c ld + r] : src[r ld + c].
// Digit s < 8 of rows [8g, 8g+8) x columns [16kb, 16kb+16) is unit
// unit + (kb * 8 + s) * groups + g of the pool, digit 8 unit
// unit / 8 + kb * groups + g of the part behind the others: two 8-row x 16-byte
// core matrices (the canonical no-swizzle K-major layout), k fast.
struct DigOperand {
  const double* src;
  long long unit;  // first unit in the pool
  int rows, k, ld, trans;
  int groups;      // ceil(rows / 8)
  int eoff;        // row exponents: exps[eoff + r]
  int koff;        // columns of the operands before it
  int pad;
};

// Which entries of a row of an operand lie how far below its maximum, for 16
// columns (a bit each): those with an exponent at most 5 (x, low half), 7 (x,
// high), 2 (y, low) and 10 (y, high) below the maximum's.  A product of entries 5
// and 7, or 2 and 10, below is at least 2^-14 of 2^ea 2^eb: x of one row and x of
// the other with its halves exchanged have a bit in common, or y and y.
// masks[unit + kb * 8 groups + r] of the operand, and the nonzero entries at the
// same place of nonzero.
using DigMask = uint2;

struct DigSeg {
  int a, b;  // operands
  double alpha;
};

// rows of an operand split by one CTA
struct DigSplit {
  int op, r0;
};

// A tile of an output block and a range of its segments.  part >= 0: the
// task stores its sum as a partial tile (128 x 64 doubles) of the scratch.
struct DigTask {
  double* C;
  long long part;
  int m, n, ldc, r0, c0;
  int seg_begin, seg_count;
  int mark;  // first of its marks (DigLaunch::flag): 8 a segment
};

struct DigReduce {
  double* C;
  long long part0;
  int m, n, ldc, r0, c0, nparts;
};

// Host lists of one launch sequence (split, products, reduction).
struct DigPlan {
  std::vector<DigOperand> ops;
  std::vector<DigSplit> splits;
  std::vector<DigSeg> segs;
  std::vector<DigTask> tasks;
  std::vector<DigReduce> reds;
  long long units = 0;    // of the digit pool
  long long scratch = 0;  // doubles of partial tiles
  int nexp = 0, nkmax = 0;
  int marks = 0;
  size_t pool_bytes() const { return (size_t)units / kDigSums * kDigSlices * kDigUnit; }
};

// Modelled SM clocks of one group by digit products and by the float64 FMA
// kernel (64 x 64 tiles, two FMAs a clock and SM), and of their longest tile.
struct DigCost {
  double digits, fma, digits_tile, fma_tile;
};
DigCost dig_cost(const GemmGroup& g, const GemmSeg* segs);

// Adds group g (its operands, shared ones once, and its tasks) to the plan.
// Groups are added whole, so a plan's numbers do not depend on where a list
// of groups is cut into plans.
class DigPlanner {
 public:
  DigPlan plan;
  void add(const GemmGroup& g, const GemmSeg* segs, int parts);
  void clear();
  size_t pool_bytes() const { return plan.pool_bytes(); }

 private:
  struct Key {
    const double* p;
    int rows, k, ld, trans;
    bool operator==(const Key& o) const {
      return p == o.p && rows == o.rows && k == o.k && ld == o.ld && trans == o.trans;
    }
  };
  struct Hash {
    size_t operator()(const Key& x) const {
      uint64_t h = (uint64_t)(uintptr_t)x.p;
      for (uint64_t v : {(uint64_t)x.rows, (uint64_t)x.k, (uint64_t)x.ld, (uint64_t)x.trans})
        h = (h ^ v) * 0x9E3779B97F4A7C15ull, h ^= h >> 29;
      return (size_t)h;
    }
  };
  std::unordered_map<Key, int, Hash> seen_;
  int operand(const double* p, int rows, int k, int ld, int trans);
};

// Partial sums a group is cut into (1: none), from its own shape alone.
int dig_parts(const GemmGroup& g, const GemmSeg* segs);

struct DigLaunch {
  const DigOperand* ops;
  const DigSplit* splits;
  const DigSeg* segs;
  const DigTask* tasks;
  const DigReduce* reds;
  int nsplits, ntasks, nreds, nops;
  unsigned char* pool;
  unsigned char* last;  // the part of the pool with the ninth digits
  double* scratch;
  int* exps;           // nexp
  DigMask* masks;      // units + 32
  uint16_t* nonzero;   // the same
  bool by_entry;       // outputs that the digits hold less well than FMAs are left out
  int* special;        // nops, and the length of `left`, zero at launch
  // A mark stands for a segment on a 32 x 32 block of a task's tile (row quarter
  // + 4 column half): flag 1 when products of it are left out, then bit c of
  // miss[32 mark + r] says that the product of row r and column c is.
  unsigned char* flag;
  uint32_t* miss;
  int* left;           // 8 task + block of the blocks with marks set, in any order
  int* err;            // host-mapped flag, set when a bounded wait ran out
  unsigned long long wait_ns;  // bound of every wait (0: its first probe)
  int sms;
};
void dig_launch(const DigLaunch& L, cudaStream_t st);

}  // namespace dmrg
