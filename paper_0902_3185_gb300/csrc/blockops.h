// Launchers of the block kernels of the DMRG step around the product:
// Kronecker growth of block operators, batched float64 GEMMs (density
// matrices, basis changes), batched symmetric eigensolves and the global
// top-m selection of density-matrix eigenvalues.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "devpool.h"

namespace dmrg {

// dst[i][j] += scale * S(i, j) for a rows x cols destination rectangle;
// S(i, j) = src[i*ld_src + j] (trans 0), src[j*ld_src + i] (trans 1), or
// the identity (src == nullptr).  Destinations of one launch must not overlap.
struct ScatJob {
  const double* src;
  double* dst;
  int32_t rows, cols, ld_src, ld_dst, trans, pad;
  double scale;
};
void launch_scatter(const std::vector<ScatJob>& jobs, cudaStream_t st);

// C = alpha op(A) op(B) + beta C for every job (op = transpose when t* = 1):
// op(A) is M x K (A row-major with leading dimension lda), op(B) K x N.
// beta = 0 does not read C.  Outputs of one launch must not overlap.
struct GemmJob {
  const double* A;
  const double* B;
  double* C;
  int32_t M, N, K, lda, ldb, ldc, ta, tb;
  double alpha, beta;
};
void launch_gemm(const std::vector<GemmJob>& jobs, cudaStream_t st);

// Eigen-decomposition of symmetric n x n matrices by cyclic Jacobi rotations
// (a thread-block cluster per matrix, or one block): w (n) in decreasing order,
// V (n x n row-major, column j the eigenvector of w[j]).  A is not modified.  work: 2 n (n + 1) doubles of
// device memory per job whose n exceeds the shared-memory limit (else unused).
struct EigJob {
  const double* A;
  double* V;
  double* w;
  double* work;
  int32_t n, pad;
};
constexpr int EIG_SMEM_MAX_N = 110;  // A and V in shared memory up to this size
constexpr int EIG_CLUSTER = 16;      // blocks of a cluster, at most
// Blocks per cluster for a list of matrices: the float64 work of a round, 3 n^2
// cycles of one SM, against the cluster's barriers; and half as many where the
// list is long enough (twenty of the widest's work) that clusters take turns
// and two of 8 fit where one of 16 does.  16 / 8 blocks, ms: 24 matrices of n =
// 130 16.9 / 15.2, of 200 52 / 42; 50 of 111 27 / 12, of 160 39 / 30, of 200 88 / 83; 100 of
// 130 51 / 40, of 200 160 / 125; but 10 of 130 11.2 / 11.9, of 200 26 / 29, and 50 of 250 148 /
// 180 (one block of 8's shared memory fills an SM from about 210 on).
inline int eig_cluster_blocks(const std::vector<int>& sizes) {
  int n = 0;
  for (int s : sizes) n = s > n ? s : n;
  if (n <= 64) return 8;
  if (n <= EIG_SMEM_MAX_N || n > 208) return EIG_CLUSTER;
  double work = 0.0;
  for (int s : sizes) work += (double)s * s * s;
  return work >= 20.0 * n * n * n ? 8 : EIG_CLUSTER;
}
// Whether matrices of these sizes (up to EIG_SMEM_MAX_N) are faster one per
// cluster, or one per block.  One block takes longer for a wide matrix, but
// hundreds of them run side by side; clusters take turns.  Modelled times (ms)
// of both, from measured ones:
//   one matrix, one block / cluster: n = 16 0.37 / 0.54, 32 1.07 / 1.21, 40 1.86 /
//   1.59, 64 5.2 / 2.7, 65 5.5 / 3.0, 80 9.3 / 3.8, 110 23.6 / 5.9 (the square roots and
//   divisions of a round are most of a small one);
//   24 matrices: 33 1.6 / 1.7, 40 2.2 / 2.0, 64 5.5 / 3.2, 110 24 / 10;
//   64 wide: 60 matrices 5.6 / 4.2, 80 5.7 / 7.0; 65 wide: 40 6.1 / 7.3; 80 wide: 40
//   10.1 / 10.0, 60 10.2 / 11.4;
//   150 matrices: 33 2.2 / 4.9, 64 6.0 / 10.5, 65 6.6 / 20.5, 110 25 / 45; 600: 64 20 / 34,
//   80 36 / 101.
inline bool eig_clusters_pay(const std::vector<int>& sizes) {
  int n = 0;
  for (int s : sizes) n = s > n ? s : n;
  if (n <= 32) return false;
  const bool wide = eig_cluster_blocks(sizes) == EIG_CLUSTER;
  const double block = 0.026 * n + 1.56e-5 * n * n * n;                       // the widest, alone in its block
  const double cluster = wide ? 0.0346 * n + 1.7e-4 * n * n : 0.0415 * n;     // alone in its cluster
  double share = 0.0;  // the clusters' time when they keep the device busy
  for (int s : sizes) share += (wide ? 0.0028 : 0.0013) * s;
  const double few = cluster + 0.4 * share;
  return (few > share ? few : share) < block + 0.1 * share;
}
void launch_eig(const std::vector<EigJob>& jobs, cudaStream_t st);

// Global selection of the m largest density-matrix eigenvalues over n
// candidates (lam, sector, index within the sector in decreasing order):
// values within tie_tol of their neighbour in decreasing order form one
// cluster, and the order is (cluster, sector, index); the first m are kept.
// keep[i] = 1 for kept candidates; out[0] = sum of the discarded eigenvalues,
// out[1] = the m-th value minus the (m+1)-th (the gap at the cut; 0 if
// n <= m).  scratch: 4 n int32 + n double of device memory.
void launch_select(const double* lam, const int32_t* sec, const int32_t* idx, int32_t n, int32_t m,
                   double tie_tol, int32_t* keep, double* out, int32_t* scratch_i, double* scratch_d,
                   cudaStream_t st);

// x[i] = uniform(-1, 1) from splitmix64 of (seed, i): the Lanczos start
// vector of a DMRG step (any vector with a component along the ground state)
void launch_start_vector(double* x, int64_t n, uint64_t seed, cudaStream_t st);

}  // namespace dmrg
