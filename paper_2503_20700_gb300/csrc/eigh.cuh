// Float64 eigensolver of a batch of symmetric matrices (the density-matrix
// sectors of a decimation, two-orbital density matrices, the Fiedler problem).
//
//   n <= kEighSmall   cyclic Jacobi in shared memory, one CTA per matrix
//   larger            Householder tridiagonalisation on a group of CTAs per
//                     matrix, divide and conquer of the tridiagonal matrix
//                     (Cuppen, Numer. Math. 36 (1981) 177; secular equation by
//                     Bunch, Nielsen and Sorensen, Numer. Math. 31 (1978) 31;
//                     eigenvectors of the recomputed rank-one update by Gu and
//                     Eisenstat, SIAM J. Matrix Anal. Appl. 16 (1995) 172) with
//                     its products on the grouped GEMM, and the reflectors
//                     applied to the eigenvectors.
// Both work on the matrix divided by a power of two that brings its largest
// entry to about one.
#pragma once
#include <cuda_runtime.h>

#include <vector>

#include "backend.hpp"

namespace dmrg {

constexpr int kEighSmall = 32;  // largest matrix of the Jacobi kernel
constexpr int kEighLeaf = 16;   // largest tridiagonal block that is not divided

// One matrix of the divide-and-conquer path.  Arrays of n start at the
// matrix's offset (the sum of the sizes before it) in the flat arrays of
// DcArrays.
struct DcMatrix {
  double* A;        // n x n; row k keeps reflector k (columns k + 1 ...)
  double* w;        // eigenvalues, descending
  double* V;        // eigenvectors as rows; holds the rank-one update's until the end
  double* B[2];     // eigenvectors of T (rows) before and after a level of merges
  double* xch;      // 8 n: what the CTAs of a group exchange, zero at launch
  unsigned* peak;   // largest entry of each CTA's rows
  unsigned* bar;    // arrivals of the group barrier, zero at launch
  int n, off;
  int g, cta0;      // CTAs of the group, the first one
  int rows_in_smem;
  int levels;       // of merges
};

// a leaf (n2 = 0) or a merge of [lo, lo + n1) and [lo + n1, lo + n1 + n2)
struct DcNode {
  int mat, off;     // off: DcMatrix::off + lo
  int lo, n1, n2;
  int first;        // sum of the sizes of the nodes before it in its list
};

struct DcRot {
  int p, q;         // rows of the children's eigenvectors, relative to lo
  double c, s;
};

// flat arrays over all matrices (length: the sum of the sizes)
struct DcArrays {
  double *d, *e, *tau;      // T, and the reflectors' factors c
  double* scale;            // per matrix
  double* val;              // eigenvalues of the current nodes, ascending
  double *dl, *zl;          // poles and z of a merge: kept ones, then deflated values
  double *mu, *zhat, *ninv; // root j: val = dl[org[j]] + mu[j]; 1 / norm of its vector
  int *org, *pos, *inv;     // pos: row of item t; inv: item of rank c
  DcRot* rot;
  int *count;               // 2 per position of a node's start: kept poles, rotations
  double* rho;              // per node start
  double* wide;             // of matrices beyond shared memory (tridiag_wide)
};

// Host plan of a batch: nodes of the leaves and of every level of merges.
struct DcPlan {
  std::vector<DcNode> leaves;
  std::vector<std::vector<DcNode>> merges;  // [level]
};
// levels of merges of an n x n tridiagonal matrix
int dc_levels(int n);
// n: sizes in descending order
DcPlan dc_plan(const std::vector<int>& n);

// rows of a CTA of a group of g (interleaved) that shared memory has room for
bool tridiag_rows_fit(int n, int g);
int tridiag_max_ctas(int sms);  // co-resident CTAs of the cooperative launch
// doubles of DcArrays::wide for matrices of at most n, `total` the sum of the
// sizes, in launches of at most `ctas`
size_t tridiag_wide(int n, int total, int ctas);

void eigh_small_launch(const EighTask* tasks, int count, cudaStream_t st);
// matrices [m0, m0 + count) of the list, ctas in all: one cooperative launch
void tridiag_launch(const DcMatrix* mats, int m0, int count, int ctas, DcArrays ar, int* err,
                    unsigned long long wait_ns, cudaStream_t st);
void dc_leaves_launch(const DcMatrix* mats, const DcNode* nodes, int count, DcArrays ar, cudaStream_t st);
// one level of merges up to the eigenvectors of the rank-one updates (in
// DcMatrix::V); positions: sum of the nodes' sizes, largest: the largest
void dc_merge_launch(const DcMatrix* mats, const DcNode* nodes, int count, int positions, int largest, int level,
                     DcArrays ar, cudaStream_t st);
void dc_back_launch(const DcMatrix* mats, int count, int rows, int largest, DcArrays ar, cudaStream_t st);

}  // namespace dmrg
