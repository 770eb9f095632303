// Block kernels of the DMRG step around the superblock product (paper
// Sec. 3.1 and Sec. 3.3: growth S' = S (x) site with the operators
// re-expressed in the product basis, the reduced density matrices
// rho_S = Psi Psi^T and rho_E = Psi^T Psi of Eqs. rhoSystem / rhoEnviron,
// their eigenvectors, the choice of the m most probable states, and the
// change of basis W^T O W of Eq. transformation).
//
// All of it is float64: the density-matrix eigenvectors decide the basis of
// every later step, and the paper's method keeps it exact to rounding.
// Sizes are small (sector blocks of a few hundred at most), so the kernels
// favour simple, bounded loops over peak throughput; the step's cost stays in
// the Lanczos solve.

#include <algorithm>
#include <cmath>
#include <cstring>
#include <stdexcept>
#include <string>

#include <cooperative_groups.h>

#include "blockops.h"

namespace dmrg {

namespace {

// The job lists of one launch on the device: one allocation (from the calling
// thread's pool, else on the stream) and one copy for both arrays, released in
// stream order after the launch.
struct Upload {
  char* p = nullptr;
  size_t bytes = 0;
  cudaStream_t st;
  DevPool* pool;
  template <class A, class B>
  Upload(const std::vector<A>& a, const std::vector<B>& b, const A** da, const B** db, cudaStream_t s)
      : st(s), pool(DevPool::current()) {
    const size_t na = (a.size() * sizeof(A) + 15) & ~(size_t)15, nb = b.size() * sizeof(B);
    bytes = std::max<size_t>(na + nb, 16);
    std::vector<char> host(bytes);
    if (!a.empty()) memcpy(host.data(), a.data(), a.size() * sizeof(A));
    if (!b.empty()) memcpy(host.data() + na, b.data(), nb);
    cudaError_t e = cudaSuccess;
    if (pool) p = static_cast<char*>(pool->get(bytes));
    else e = cudaMallocAsync(reinterpret_cast<void**>(&p), bytes, st);
    if (e != cudaSuccess) throw std::runtime_error(std::string("cudaMallocAsync: ") + cudaGetErrorString(e));
    e = cudaMemcpyAsync(p, host.data(), bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) {
      release();
      throw std::runtime_error(std::string("cudaMemcpyAsync: ") + cudaGetErrorString(e));
    }
    *da = reinterpret_cast<const A*>(p);
    *db = reinterpret_cast<const B*>(p + na);
  }
  ~Upload() { release(); }
  void release() {
    if (!p) return;
    if (pool) pool->put(p, bytes);
    else cudaFreeAsync(p, st);
    p = nullptr;
  }
  Upload(const Upload&) = delete;
  Upload& operator=(const Upload&) = delete;
};

void check_launch(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) throw std::runtime_error(std::string(what) + ": " + cudaGetErrorString(e));
}

struct Tile {
  int32_t job, i0, j0, pad;
};

}  // namespace

// ------------------------------------------------------------------ scatter
// One 32 x 32 destination tile per block (32 x 8 threads); a transposed
// source goes through shared memory so that both the read and the write run
// along rows.
__global__ void __launch_bounds__(256) k_scatter(const ScatJob* __restrict__ jobs, const Tile* __restrict__ tiles) {
  __shared__ double t[32][33];
  const Tile tl = tiles[blockIdx.x];
  const ScatJob jb = jobs[tl.job];
  const int tx = threadIdx.x, ty = threadIdx.y;
  if (jb.src && jb.trans) {
    for (int r = ty; r < 32; r += 8) {
      const int j = tl.j0 + r, i = tl.i0 + tx;
      t[r][tx] = (j < jb.cols && i < jb.rows) ? jb.src[(int64_t)j * jb.ld_src + i] : 0.0;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
      const int i = tl.i0 + r, j = tl.j0 + tx;
      if (i < jb.rows && j < jb.cols) jb.dst[(int64_t)i * jb.ld_dst + j] += jb.scale * t[tx][r];
    }
  } else {
    for (int r = ty; r < 32; r += 8) {
      const int i = tl.i0 + r, j = tl.j0 + tx;
      if (i < jb.rows && j < jb.cols) {
        const double v = jb.src ? jb.src[(int64_t)i * jb.ld_src + j] : (i == j ? 1.0 : 0.0);
        jb.dst[(int64_t)i * jb.ld_dst + j] += jb.scale * v;
      }
    }
  }
}

void launch_scatter(const std::vector<ScatJob>& jobs, cudaStream_t st) {
  std::vector<Tile> tiles;
  for (size_t q = 0; q < jobs.size(); ++q)
    for (int i0 = 0; i0 < jobs[q].rows; i0 += 32)
      for (int j0 = 0; j0 < jobs[q].cols; j0 += 32) tiles.push_back({(int32_t)q, i0, j0, 0});
  if (tiles.empty()) return;
  const ScatJob* dj;
  const Tile* dt;
  const Upload up(jobs, tiles, &dj, &dt, st);
  k_scatter<<<(unsigned)tiles.size(), dim3(32, 8), 0, st>>>(dj, dt);
  check_launch("k_scatter");
}

// ------------------------------------------------------------------- gemm
// 64 x 64 output tile per block, 256 threads of 4 x 4 outputs each, K in
// chunks of 16 through shared memory (operands loaded along their
// contiguous index whatever the transpose).
__global__ void __launch_bounds__(256) k_gemm(const GemmJob* __restrict__ jobs, const Tile* __restrict__ tiles) {
  __shared__ double As[16][65];
  __shared__ double Bs[16][65];
  const Tile tl = tiles[blockIdx.x];
  const GemmJob jb = jobs[tl.job];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = tl.i0, n0 = tl.j0;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < jb.K; k0 += 16) {
    for (int e = tid; e < 1024; e += 256) {
      int mm, kk;
      if (jb.ta) { kk = e >> 6; mm = e & 63; } else { mm = e >> 4; kk = e & 15; }
      const int m = m0 + mm, k = k0 + kk;
      double v = 0.0;
      if (m < jb.M && k < jb.K) v = jb.ta ? jb.A[(int64_t)k * jb.lda + m] : jb.A[(int64_t)m * jb.lda + k];
      As[kk][mm] = v;
    }
    for (int e = tid; e < 1024; e += 256) {
      int nn, kk;
      if (jb.tb) { nn = e >> 4; kk = e & 15; } else { kk = e >> 6; nn = e & 63; }
      const int n = n0 + nn, k = k0 + kk;
      double v = 0.0;
      if (n < jb.N && k < jb.K) v = jb.tb ? jb.B[(int64_t)n * jb.ldb + k] : jb.B[(int64_t)k * jb.ldb + n];
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= jb.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx + 16 * j;
      if (n >= jb.N) continue;
      double* c = jb.C + (int64_t)m * jb.ldc + n;
      *c = jb.beta != 0.0 ? fma(jb.alpha, acc[i][j], jb.beta * *c) : jb.alpha * acc[i][j];
    }
  }
}

void launch_gemm(const std::vector<GemmJob>& jobs, cudaStream_t st) {
  std::vector<Tile> tiles;
  for (size_t q = 0; q < jobs.size(); ++q) {
    const GemmJob& j = jobs[q];
    if (j.M <= 0 || j.N <= 0) continue;
    for (int m0 = 0; m0 < j.M; m0 += 64)
      for (int n0 = 0; n0 < j.N; n0 += 64) tiles.push_back({(int32_t)q, m0, n0, 0});
  }
  if (tiles.empty()) return;
  const GemmJob* dj;
  const Tile* dt;
  const Upload up(jobs, tiles, &dj, &dt, st);
  k_gemm<<<(unsigned)tiles.size(), 256, 0, st>>>(dj, dt);
  check_launch("k_gemm");
}

// ---------------------------------------------------------------- eigen
// Cyclic Jacobi (Golub & Van Loan, Sec. 8.5) with the round-robin ordering:
// in each of the N2 - 1 rounds of a sweep the N2 / 2 rotations are disjoint,
// so all of them are applied at once -- rows p, q of A for every pair, then
// columns p, q of A and of V -- as A <- J^T A J, V <- V J.  The rotation that
// zeroes a_pq: tau = (a_qq - a_pp) / (2 a_pq), t = sign(tau) / (|tau| +
// sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c.  A rotation is skipped
// when |a_pq| <= 4 eps |A|_F (threshold Jacobi: rounding leaves off-diagonal
// elements near eps |A|, so a tighter test would never pass), and the sweeps
// stop after one without a rotation (at most 40).  The eigenvalues are then
// accurate to a few eps |A| in absolute terms, as a LAPACK solver's.
constexpr int EIG_THREADS = 256;
constexpr int EIG_MAX_N = 4096;

__device__ __forceinline__ double eig_block_sum(double v, double* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
  return t;
}

__device__ __forceinline__ int rr_player(int slot, int r, int n2) {
  return slot == 0 ? 0 : 1 + (slot - 1 + r) % (n2 - 1);
}

__global__ void __launch_bounds__(EIG_THREADS) k_eig(const EigJob* __restrict__ jobs) {
  extern __shared__ double sm[];
  __shared__ double red[EIG_THREADS / 32];
  const EigJob jb = jobs[blockIdx.x];
  const int n = jb.n;
  if (n <= 0) return;
  const int ld = n + 1;
  const int n2 = (n + 1) & ~1;
  const int np = n2 / 2;
  const bool in_smem = n <= EIG_SMEM_MAX_N;
  double* a = in_smem ? sm : jb.work;
  double* v = in_smem ? sm + (size_t)n * ld : jb.work + (size_t)n * ld;
  double* base = in_smem ? sm + (size_t)2 * n * ld : sm;
  double* cs = base;           // [np]
  double* sn = base + np;      // [np]
  int* pp = reinterpret_cast<int*>(base + 2 * np);  // [np]
  int* qq = pp + np;                                 // [np]
  int* rank = qq + np;                               // [n]
  const int tid = threadIdx.x;
  for (int e = tid; e < n * n; e += EIG_THREADS) {
    const int i = e / n, j = e % n;
    a[i * ld + j] = jb.A[(int64_t)i * n + j];
    v[i * ld + j] = i == j ? 1.0 : 0.0;
  }
  __syncthreads();
  if (n > 1) {
    double fro = 0.0;
    for (int e = tid; e < n * n; e += EIG_THREADS) {
      const double x = a[(e / n) * ld + e % n];
      fro = fma(x, x, fro);
    }
    const double thr = 4.0 * 2.220446049250313e-16 * sqrt(eig_block_sum(fro, red));
    for (int sweep = 0; sweep < 40; ++sweep) {
      double rot = 0.0;  // rotations applied by this thread in the sweep
      for (int r = 0; r < n2 - 1; ++r) {
        for (int k = tid; k < np; k += EIG_THREADS) {
          int p = rr_player(k, r, n2), q = rr_player(n2 - 1 - k, r, n2);
          if (p > q) { const int t = p; p = q; q = t; }
          double c = 1.0, s = 0.0;
          if (q < n) {
            const double apq = a[p * ld + q];
            if (fabs(apq) > thr) {
              const double tau = (a[q * ld + q] - a[p * ld + p]) / (2.0 * apq);
              double t;
              if (fabs(tau) > 1e150) t = 0.5 / tau;
              else t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
              c = 1.0 / sqrt(1.0 + t * t);
              s = t * c;
              rot += 1.0;
            }
          }
          pp[k] = p;
          qq[k] = q;
          cs[k] = c;
          sn[k] = s;
        }
        __syncthreads();
        for (int e = tid; e < np * n; e += EIG_THREADS) {  // rows p, q
          const int k = e / n, j = e % n;
          const double s = sn[k];
          if (s == 0.0) continue;
          const double c = cs[k];
          const int p = pp[k], q = qq[k];
          const double x = a[p * ld + j], y = a[q * ld + j];
          a[p * ld + j] = c * x - s * y;
          a[q * ld + j] = s * x + c * y;
        }
        __syncthreads();
        for (int e = tid; e < np * n; e += EIG_THREADS) {  // columns p, q of A and V
          const int k = e / n, i = e % n;
          const double s = sn[k];
          if (s == 0.0) continue;
          const double c = cs[k];
          const int p = pp[k], q = qq[k];
          const double x = a[i * ld + p], y = a[i * ld + q];
          a[i * ld + p] = c * x - s * y;
          a[i * ld + q] = s * x + c * y;
          const double xv = v[i * ld + p], yv = v[i * ld + q];
          v[i * ld + p] = c * xv - s * yv;
          v[i * ld + q] = s * xv + c * yv;
        }
        __syncthreads();
      }
      if (eig_block_sum(rot, red) == 0.0) break;  // the same sum in every thread
    }
  }
  // decreasing order (ties by index)
  for (int i = tid; i < n; i += EIG_THREADS) {
    const double wi = a[i * ld + i];
    int rk = 0;
    for (int j = 0; j < n; ++j) {
      const double wj = a[j * ld + j];
      rk += (wj > wi) || (wj == wi && j < i);
    }
    rank[i] = rk;
  }
  __syncthreads();
  for (int i = tid; i < n; i += EIG_THREADS) jb.w[rank[i]] = a[i * ld + i];
  for (int e = tid; e < n * n; e += EIG_THREADS) {
    const int row = e / n, i = e % n;
    jb.V[(int64_t)row * n + rank[i]] = v[row * ld + i];
  }
}

// The same cyclic Jacobi on a thread-block cluster, for matrices whose columns
// fit the cluster's shared memory.
//
// What bounds it: one SM issues 2 float64 operations per clock, and a round
// costs 6 n^2 of them (rows and columns of A, columns of V), so the round is
// spread over the cluster's SMs; then the barriers between its steps count.
// The round-robin ordering is played as a tournament: block c of the cluster
// keeps a run of neighbouring pair slots, the columns of A and V of both
// players of each.  Given all rotations of the round, everything is local to
// a column pair: the row rotations act within a column, then the pair's own
// rotation mixes its two columns (and those of V).  Between rounds the players
// move on by one slot: inside a block that is a change of a table, and two
// columns cross to the neighbouring blocks (distributed shared memory, into a
// spare column there).  So a round has two cluster barriers: after A's columns
// have moved, and after the next round's rotations are published to every
// block; V, which no rotation depends on, is rotated between the two, beside
// the square roots and divisions of those rotations.
// Rotation order and arithmetic are those of k_eig (every element sees the
// same operations in the same order).
//
// Measured against one block with A and V in shared memory (up to n = 110) and
// a 16-block cluster with rows dealt to the blocks and three barriers a round
// (above): one matrix of n = 48 2.79 -> 2.05 ms, 64 5.35 -> 2.8, 80 9.88 -> 3.6,
// 110 24.7 -> 6.2, 300 66.7 -> 58 ms; 24 of n = 110 24.8 -> 10 ms.  At n = 300 the
// float64 unit of the cluster's SMs is 43 % busy (a sweep is 18 million cycles
// of it per 1000 rounds, 9 to 10 sweeps); 512 threads per block were faster
// for one wide matrix (51 ms) but slower for many (24 of n = 110 15.5 ms).
// x != 0 by its bits (a float64 compare runs on the float64 unit)
__device__ __forceinline__ bool nonzero(double x) {
  return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) != 0;
}

__host__ __device__ inline int eig_active_blocks(int np, int C) { return np / 2 < 1 ? 1 : (np / 2 < C ? np / 2 : C); }

constexpr int EIGC_THREADS = 256, EIGC_WARPS = EIGC_THREADS / 32;

__global__ void __launch_bounds__(EIGC_THREADS) k_eig_cluster(const EigJob* __restrict__ jobs) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ double sm[];
  __shared__ double red[EIGC_WARPS];
  __shared__ double sums[1];
  const int C = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  const EigJob jb = jobs[blockIdx.x / C];
  const int n = jb.n;
  const int n2 = (n + 1) & ~1;
  const int np = n2 / 2;
  // this block's pairs: slots k0 .. k0 + m - 1 of the top row and the ones facing them
  const int Ca = eig_active_blocks(np, C);
  const int base = np / Ca, rem = np % Ca, mmax = base + (rem > 0);
  const int m = rank < Ca ? base + (rank < rem) : 0;
  const int k0 = rank < Ca ? rank * base + min(rank, rem) : np;
  const int ncol = 2 * mmax + 2;
  double2* allp = reinterpret_cast<double2*>(sm);     // [2][np] (c, s) of this round and the next
  double* a = sm + 4 * np;                            // [ncol][n] columns of A
  double* v = a + (size_t)ncol * n;                   // [ncol][n] columns of V
  double* dg = v + (size_t)ncol * n;                  // [n] diagonal (final ordering)
  int* rk = reinterpret_cast<int*>(dg + n);           // [n]
  int* top = rk + n;                                  // [2][mmax] column of each top slot, this round and the next
  int* bot = top + 2 * mmax;                          // [2][mmax] of the slot facing it
  int* spare = bot + 2 * mmax;                        // [2][2] where a column from the right, the left goes
  short2* rows = reinterpret_cast<short2*>(spare + 4);  // [2][np] (p, q) of each pair, this round and the next
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int e = tid; e < 2 * m * n; e += EIGC_THREADS) {
    const int i = e / (2 * m), lc = e % (2 * m);
    const int j = lc < m ? k0 + lc : n2 - 1 - (k0 + lc - m);  // the player of a slot before the first round
    if (j < n) {
      a[(size_t)lc * n + i] = jb.A[(int64_t)i * n + j];
      v[(size_t)lc * n + i] = i == j ? 1.0 : 0.0;
    }
  }
  for (int kk = tid; kk < m; kk += EIGC_THREADS) {
    top[kk] = kk;
    bot[kk] = m + kk;
  }
  if (tid == 0) {
    spare[0] = 2 * m;
    spare[1] = 2 * m + 1;
  }
  // |A|_F^2 by the first EIG_THREADS threads, summed as in k_eig
  double fro = 0.0;
  if (tid < EIG_THREADS)
    for (int e = tid; e < n * n; e += EIG_THREADS) {
      const double x = jb.A[e];
      fro = fma(x, x, fro);
    }
  const double thr = 4.0 * 2.220446049250313e-16 * sqrt(eig_block_sum(fro, red));
  // the pairs of round r, and its rotations from the columns in place (tables
  // tp, bt), published to every block
  double rot = 0.0;  // rotations this thread computed
  auto rotations = [&](int r, const int* tp, const int* bt, double2* out, short2* pq) {
    for (int k = tid; k < np; k += EIGC_THREADS) {
      const int pt = rr_player(k, r, n2), pb = rr_player(n2 - 1 - k, r, n2);
      pq[k] = make_short2((short)min(pt, pb), (short)max(pt, pb));
    }
    for (int kk = tid; kk < m; kk += EIGC_THREADS) {
      const int k = k0 + kk;
      const int pt = rr_player(k, r, n2), pb = rr_player(n2 - 1 - k, r, n2);
      const int p = min(pt, pb), q = max(pt, pb);
      double c = 1.0, s = 0.0;
      if (q < n) {
        const double* ap = a + (size_t)(pt < pb ? tp[kk] : bt[kk]) * n;
        const double* aq = a + (size_t)(pt < pb ? bt[kk] : tp[kk]) * n;
        const double apq = aq[p];
        if (fabs(apq) > thr) {
          const double tau = (aq[q] - ap[p]) / (2.0 * apq);
          double t;
          if (fabs(tau) > 1e150) t = 0.5 / tau;
          else t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
          c = 1.0 / sqrt(1.0 + t * t);
          s = t * c;
          rot += 1.0;
        }
      }
      const double2 cs = make_double2(c, s);
      for (int b = 0; b < Ca; ++b) cl.map_shared_rank(out, b)[k] = cs;
    }
  };
  cl.sync();
  if (n > 1) rotations(0, top, bot, allp, rows);
  cl.sync();
  int par = 0;
  for (int sweep = 0; n > 1 && sweep < 40; ++sweep) {
    double done = 0.0;  // rotations of this sweep
    for (int r = 0; r < n2 - 1; ++r) {
      const int* tp = top + par * mmax;
      const int* bt = bot + par * mmax;
      const int* sp = spare + par * 2;
      const double2* cs = allp + (size_t)par * np;
      const short2* pq = rows + (size_t)par * np;
      const int nch = (np + 31) / 32;
      for (int task = wid; task < m * nch; task += EIGC_WARPS) {  // A: a column pair's elements of 32 row pairs
        const int kk = task / nch, kr = (task - kk * nch) * 32 + lane;
        if (kr >= np) continue;
        const double2 col = cs[k0 + kk], row = cs[kr];
        const bool rcol = nonzero(col.y), rrow = nonzero(row.y);
        if (!rcol && !rrow) continue;
        const short2 own = pq[k0 + kk], rr = pq[kr];
        const bool tf = rr_player(k0 + kk, r, n2) == own.x;
        double* ap = a + (size_t)(tf ? tp[kk] : bt[kk]) * n;
        double* aq = a + (size_t)(tf ? bt[kk] : tp[kk]) * n;
        const bool hasq = own.y < n;  // else column p has no partner this round
        const int rp = rr.x, rq = rr.y;
        const bool hasr = rq < n;
        double x11 = ap[rp], x21 = hasr ? ap[rq] : 0.0;
        double x12 = hasq ? aq[rp] : 0.0, x22 = hasq && hasr ? aq[rq] : 0.0;
        if (rrow) {
          const double c = row.x, s = row.y;
          const double x = x11, y = x21;
          x11 = c * x - s * y;
          x21 = s * x + c * y;
          const double x2 = x12, y2 = x22;
          x12 = c * x2 - s * y2;
          x22 = s * x2 + c * y2;
        }
        if (rcol) {
          const double c = col.x, s = col.y;
          const double x = x11, y = x12;
          x11 = c * x - s * y;
          x12 = s * x + c * y;
          const double x2 = x21, y2 = x22;
          x21 = c * x2 - s * y2;
          x22 = s * x2 + c * y2;
        }
        ap[rp] = x11;
        if (hasr) ap[rq] = x21;
        if (hasq) {
          aq[rp] = x12;
          if (hasr) aq[rq] = x22;
        }
      }
      __syncthreads();
      // the players move on: tops down by one slot, facing slots up, around
      // the ends; the columns sent away are the next spares
      const bool left = np > 1 && rank > 0 && rank < Ca, right = np > 1 && rank < Ca - 1;
      int* nt = top + (par ^ 1) * mmax;
      int* nb = bot + (par ^ 1) * mmax;
      for (int kk = tid; kk < m; kk += EIGC_THREADS) {
        nt[kk] = k0 + kk == 0 ? tp[0] : (kk < m - 1 ? tp[kk + 1] : (right ? sp[0] : bt[m - 1]));
        nb[kk] = np == 1 ? bt[0] : (kk > 0 ? bt[kk - 1] : (left ? sp[1] : tp[1]));
      }
      if (tid == 0 && m > 0) {
        spare[(par ^ 1) * 2] = left ? tp[0] : bt[m - 1];
        spare[(par ^ 1) * 2 + 1] = right ? bt[m - 1] : tp[0];
      }
      const size_t to_left = left ? (size_t)cl.map_shared_rank(spare, rank - 1)[par * 2] * n : 0;
      const size_t to_right = right ? (size_t)cl.map_shared_rank(spare, rank + 1)[par * 2 + 1] * n : 0;
      auto move = [&](double* cols) {
        if (left) {
          double* dst = cl.map_shared_rank(cols, rank - 1) + to_left;
          const double* src = cols + (size_t)tp[0] * n;
          for (int i = tid; i < n; i += EIGC_THREADS) dst[i] = src[i];
        }
        if (right) {
          double* dst = cl.map_shared_rank(cols, rank + 1) + to_right;
          const double* src = cols + (size_t)bt[m - 1] * n;
          for (int i = tid; i < n; i += EIGC_THREADS) dst[i] = src[i];
        }
      };
      move(a);
      cl.sync();  // A's columns are where the next round wants them
      done += rot;
      rot = 0.0;
      rotations(r + 1 < n2 - 1 ? r + 1 : 0, nt, nb, allp + (size_t)(par ^ 1) * np,
                rows + (size_t)(par ^ 1) * np);
      const int nchv = (n + 31) / 32;
      for (int task = wid; task < m * nchv; task += EIGC_WARPS) {  // V, beside the next rotations
        const int kk = task / nchv, i = (task - kk * nchv) * 32 + lane;
        const double2 col = cs[k0 + kk];
        if (i >= n || !nonzero(col.y)) continue;
        const bool tf = rr_player(k0 + kk, r, n2) == pq[k0 + kk].x;
        double* vp = v + (size_t)(tf ? tp[kk] : bt[kk]) * n;
        double* vq = v + (size_t)(tf ? bt[kk] : tp[kk]) * n;
        const double c = col.x, s = col.y;
        const double xv = vp[i], yv = vq[i];
        vp[i] = c * xv - s * yv;
        vq[i] = s * xv + c * yv;
      }
      __syncthreads();
      move(v);
      par ^= 1;
      cl.sync();  // the next rotations and V's columns are everywhere
    }
    done = eig_block_sum(done, red);
    if (tid == 0) sums[0] = done;
    cl.sync();
    double all = 0.0;
    for (int b = 0; b < C; ++b) all += cl.map_shared_rank(sums, b)[0];
    cl.sync();  // read before any block writes the next one
    if (all == 0.0) break;  // every block leaves together
  }
  // decreasing order (ties by index): every block gathers the diagonal and
  // ranks it, and writes its own columns of V
  auto slot_col = [&](int lc, int& j) -> int {  // local column lc < 2 m: its index in A and its place
    j = lc < m ? k0 + lc : n2 - 1 - (k0 + lc - m);
    return lc < m ? top[par * mmax + lc] : bot[par * mmax + lc - m];
  };
  for (int lc = tid; lc < 2 * m; lc += EIGC_THREADS) {
    int j;
    const int col = slot_col(lc, j);
    if (j >= n) continue;
    const double d = a[(size_t)col * n + j];
    for (int b = 0; b < Ca; ++b) cl.map_shared_rank(dg, b)[j] = d;
  }
  cl.sync();
  if (m == 0) return;
  for (int i = tid; i < n; i += EIGC_THREADS) {
    const double wi = dg[i];
    int r2 = 0;
    for (int j = 0; j < n; ++j) r2 += (dg[j] > wi) || (dg[j] == wi && j < i);
    rk[i] = r2;
  }
  __syncthreads();
  if (rank == 0)
    for (int i = tid; i < n; i += EIGC_THREADS) jb.w[rk[i]] = dg[i];
  for (int e = tid; e < 2 * m * n; e += EIGC_THREADS) {
    const int i = e / (2 * m), lc = e % (2 * m);
    int j;
    const int col = slot_col(lc, j);
    if (j < n) jb.V[(int64_t)i * n + rk[j]] = v[(size_t)col * n + i];
  }
}

size_t eig_cluster_smem(int n, int C) {
  const size_t np = (size_t)(n + 1) / 2;
  const size_t Ca = (size_t)eig_active_blocks((int)np, C), mmax = (np + Ca - 1) / Ca;
  return (4 * np + 2 * (2 * mmax + 2) * n + n) * sizeof(double) + (n + 4 * mmax + 4 + 2 * np) * sizeof(int);
}

// largest n the cluster kernel takes (A and V in the cluster's shared memory)
constexpr int EIG_CLUSTER_MAX_N = 448;

// -1: not tried, 0: unavailable on this device, 1: available
int g_cluster_ok = -1;

// one launch, the largest matrices first; false if the device has no such clusters
bool launch_eig_cluster(std::vector<EigJob> jobs, cudaStream_t st) {
  if (jobs.empty()) return true;
  if (g_cluster_ok == 0) return false;
  std::stable_sort(jobs.begin(), jobs.end(), [](const EigJob& x, const EigJob& y) { return x.n > y.n; });
  std::vector<int> sizes;
  for (const EigJob& j : jobs) sizes.push_back(j.n);
  const int C = eig_cluster_blocks(sizes);
  size_t smem = 0;
  for (const EigJob& j : jobs) smem = std::max(smem, eig_cluster_smem(j.n, C));
  smem = (smem + 15) & ~(size_t)15;
  if (cudaFuncSetAttribute(k_eig_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(k_eig_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    g_cluster_ok = 0;
    return false;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(C * jobs.size()));
  cfg.blockDim = dim3(EIGC_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, k_eig_cluster, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    g_cluster_ok = 0;
    return false;
  }
  g_cluster_ok = 1;
  const EigJob* dj;
  const char* none;
  const Upload up(jobs, std::vector<char>(), &dj, &none, st);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_eig_cluster, dj);
  if (e != cudaSuccess) throw std::runtime_error(std::string("k_eig_cluster: ") + cudaGetErrorString(e));
  return true;
}

void launch_eig(const std::vector<EigJob>& all, cudaStream_t st) {
  if (all.empty()) return;
  // what exceeds one block's shared memory goes to the cluster kernel, up to its
  // limit and when the device runs it; smaller matrices where that is faster
  // (eig_clusters_pay), in a launch of their own: the larger ones' shared memory
  // would leave one block per SM.  The rest goes to the one-block kernel
  std::vector<EigJob> mid, small, jobs;
  for (const EigJob& j : all)
    if (j.n > 0) (j.n > EIG_CLUSTER_MAX_N ? jobs : j.n > EIG_SMEM_MAX_N ? mid : small).push_back(j);
  std::vector<int> sizes;
  for (const EigJob& j : small) sizes.push_back(j.n);
  for (std::vector<EigJob>* set : {&mid, &small})
    if ((set == &small && !eig_clusters_pay(sizes)) || !launch_eig_cluster(*set, st))
      for (const EigJob& j : *set) {
        if (j.n > EIG_SMEM_MAX_N && !j.work) throw std::logic_error("eigensolve: missing workspace");
        jobs.push_back(j);
      }
  if (jobs.empty()) return;
  size_t smem = 0;
  for (const EigJob& j : jobs) {
    if (j.n > EIG_MAX_N) throw std::logic_error("eigensolve: block larger than 4096");
    if (j.n > EIG_SMEM_MAX_N && !j.work) throw std::logic_error("eigensolve: missing workspace");
    const size_t n = (size_t)std::max(j.n, 1), np = (n + 1) / 2;
    size_t b = (np * 2) * sizeof(double) + (np * 2 + n) * sizeof(int);
    if (j.n <= EIG_SMEM_MAX_N) b += 2 * n * (n + 1) * sizeof(double);
    smem = std::max(smem, b);
  }
  smem = (smem + 15) & ~(size_t)15;
  cudaError_t e = cudaFuncSetAttribute(k_eig, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) throw std::runtime_error(std::string("k_eig smem: ") + cudaGetErrorString(e));
  const EigJob* dj;
  const char* none;
  const Upload up(jobs, std::vector<char>(), &dj, &none, st);
  k_eig<<<(unsigned)jobs.size(), EIG_THREADS, smem, st>>>(dj);
  check_launch("k_eig");
}

// -------------------------------------------------------------- selection
__device__ __forceinline__ bool key_less(double la, int sa, int ia, double lb, int sb, int ib) {
  // decreasing eigenvalue, then sector, then index
  if (la != lb) return la > lb;
  if (sa != sb) return sa < sb;
  return ia < ib;
}

// rank[i] by (-lam, sec, idx); order[rank[i]] = i
__global__ void k_sel_rank(const double* __restrict__ lam, const int32_t* __restrict__ sec,
                           const int32_t* __restrict__ idx, int n, int32_t* __restrict__ rank,
                           int32_t* __restrict__ order) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double li = lam[i];
  const int si = sec[i], ii = idx[i];
  int r = 0;
  for (int j = 0; j < n; ++j) r += key_less(lam[j], sec[j], idx[j], li, si, ii);
  rank[i] = r;
  order[r] = i;
}

// cluster id (1-based) of every candidate: in decreasing order, a new cluster
// starts where the value drops by more than tie_tol from its predecessor
__global__ void __launch_bounds__(1024) k_sel_cluster(const double* __restrict__ lam, const int32_t* __restrict__ order,
                                                      const int32_t* __restrict__ rank, int n, double tie_tol,
                                                      int32_t* __restrict__ cl_sorted, int32_t* __restrict__ cl) {
  __shared__ int32_t cnt[1024];
  const int tid = threadIdx.x;
  const int per = (n + 1023) / 1024;
  const int b = min(n, tid * per), e = min(n, b + per);
  auto flag = [&](int r) { return r == 0 || (lam[order[r - 1]] - lam[order[r]] > tie_tol); };
  int c = 0;
  for (int r = b; r < e; ++r) c += flag(r);
  cnt[tid] = c;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {  // inclusive scan
    const int add = tid >= o ? cnt[tid - o] : 0;
    __syncthreads();
    cnt[tid] += add;
    __syncthreads();
  }
  int id = cnt[tid] - c;
  for (int r = b; r < e; ++r) {
    id += flag(r);
    cl_sorted[r] = id;
  }
  __syncthreads();
  for (int i = tid; i < n; i += 1024) cl[i] = cl_sorted[rank[i]];
}

// final rank by (cluster, sec, idx); keep the first m
__global__ void k_sel_keep(const int32_t* __restrict__ cl, const int32_t* __restrict__ sec,
                           const int32_t* __restrict__ idx, int n, int m, int32_t* __restrict__ keep,
                           int32_t* __restrict__ order2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int ci = cl[i], si = sec[i], ii = idx[i];
  int r = 0;
  for (int j = 0; j < n; ++j) {
    const int cj = cl[j], sj = sec[j];
    r += cj < ci || (cj == ci && (sj < si || (sj == si && idx[j] < ii)));
  }
  keep[i] = r < m;
  order2[r] = i;
}

// discarded weight (fixed-order block sum) and the gap at the cut
__global__ void __launch_bounds__(256) k_sel_stats(const double* __restrict__ lam, const int32_t* __restrict__ keep,
                                                   const int32_t* __restrict__ order2, int n, int m,
                                                   double* __restrict__ out) {
  __shared__ double red[8];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256)
    if (!keep[i]) s += lam[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    out[0] = t;
    out[1] = (m >= 1 && m < n) ? lam[order2[m - 1]] - lam[order2[m]] : 0.0;
  }
}

void launch_select(const double* lam, const int32_t* sec, const int32_t* idx, int32_t n, int32_t m, double tie_tol,
                   int32_t* keep, double* out, int32_t* scratch_i, double* scratch_d, cudaStream_t st) {
  (void)scratch_d;
  if (n <= 0) {
    cudaMemsetAsync(out, 0, 2 * sizeof(double), st);
    return;
  }
  int32_t* rank = scratch_i;
  int32_t* order = scratch_i + n;
  int32_t* cl_sorted = scratch_i + 2 * (size_t)n;
  int32_t* cl = scratch_i + 3 * (size_t)n;
  const unsigned g = (unsigned)((n + 255) / 256);
  k_sel_rank<<<g, 256, 0, st>>>(lam, sec, idx, n, rank, order);
  k_sel_cluster<<<1, 1024, 0, st>>>(lam, order, rank, n, tie_tol, cl_sorted, cl);
  // order is free again: it receives the final order
  k_sel_keep<<<g, 256, 0, st>>>(cl, sec, idx, n, m, keep, order);
  k_sel_stats<<<1, 256, 0, st>>>(lam, keep, order, n, m, out);
  check_launch("select");
}

// ----------------------------------------------------------- start vector
// splitmix64 (Steele, Lea and Flood, 2014): the state advances by the golden
// ratio increment and is finalised by two xor-shift-multiply rounds
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_start(double* __restrict__ x, int64_t n, uint64_t seed) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t z = splitmix64(seed * 0xD1B54A32D192ED03ull + (uint64_t)i);
    x[i] = 2.0 * ((double)(z >> 11) * 0x1.0p-53) - 1.0;
  }
}

void launch_start_vector(double* x, int64_t n, uint64_t seed, cudaStream_t st) {
  if (n <= 0) return;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 152 * 8);
  k_start<<<(unsigned)blocks, 256, 0, st>>>(x, n, seed);
  check_launch("k_start");
}

}  // namespace dmrg
