// Internal types of the superblock library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <string>
#include <vector>

#include "dmrg_gb300.h"

namespace dmrg {

// ---------------------------------------------------------------- FP64 path
// Buffers a task can address.  Offsets are in elements, so one task list
// serves every call whatever the caller's pointers are.
enum BufId : int32_t { BUF_X = 0, BUF_Y = 1, BUF_T = 2, BUF_OPS = 3, BUF_G = 4, NBUF = 5 };

struct Bufs {
  double* p[NBUF];
};

// One product L (M x K) * R (K x N) added into the tile, for batch member b:
// the operands start at l_off + b l_bs and r_off + b r_bs (stride 0: the
// operator blocks, shared by all members).  scale: the coefficient of the
// member's `term` multiplies L (1), R (2) or nothing (0).
struct SegF64 {
  int64_t l_off, r_off;
  int64_t l_bs, r_bs;
  int32_t l_buf, r_buf;
  int32_t ldl, ldr;
  int32_t K;
  int32_t l_trans;  // 0: L(m,k) = X[m*ldl + k]; 1: L(m,k) = X[k*ldl + m]
  int32_t r_trans;  // 0: R(k,n) = X[k*ldr + n]; 1: R(k,n) = X[n*ldr + k]
  int32_t term, scale;
  int32_t pad;
};

// One output tile C[m0:m0+8*ni, n0:n0+8*nj] of an M x N matrix (ni, nj in 1..2,
// chosen per output), for every batch member b at c_off + b c_bs.  Its
// segments form two groups, each summed by itself, then added.
enum TileMode : int32_t { TM_STORE = 0, TM_DOT = 2, TM_STORE_DOTS = 3 };
struct TileF64 {
  int64_t c_off, c_bs;
  int32_t c_buf, ldc;
  int32_t M, N, m0, n0;
  int32_t seg_begin, seg_mid, seg_end;
  int32_t mode;     // TM_STORE: C = acc (C += acc when the launch accumulates); TM_DOT: sum(acc .* C);
                    // TM_STORE_DOTS: C = sum over segments of c(member, term) * seg_acc, and per segment
                    // sum(seg_acc .* X) at the same offset of BUF_X
  int32_t shape;    // ni | nj << 8
  int32_t dot_base; // TM_STORE_DOTS: index of the tile's first segment among all (tile, segment) of the list
};

struct TaskListF64 {
  SegF64* d_segs = nullptr;
  int32_t n_outs = 0;
  TileF64* d_outs = nullptr;   // descriptors of the outputs, in the order of their tiles
  int32_t* d_first = nullptr;  // first tile of every output (+ end)
  TileF64* d_tiles = nullptr;
  bool wide = false, wide_df = false;  // tiles up to 24 wide (else 16), float64 and double-float
  int64_t n_tiles = 0;  // per member: a launch has n_tiles * batch blocks, block tile * batch + member
  // the same outputs cut for double-float arithmetic (tiles made at the first such product)
  TileF64* d_outs_df = nullptr;
  int32_t* d_first_df = nullptr;
  TileF64* d_tiles_df = nullptr;
  int64_t n_tiles_df = 0;
};

// dot partials per (tile, member), or per (tile, segment, member): one per warp of a block
constexpr int SEG_DOT_PARTS = 2;

// The partials of a dot list by term.  An item is a (tile, segment) of the list
// (a tile of a TM_DOT list); item i of member b has the partials
// (i * batch + b) * SEG_DOT_PARTS + part.  A run: the items of one output and
// segment, item + u stride for its tiles u, elements first .. end - 1 of its
// term's list.
struct DotRun {
  int32_t item, stride, first, end;
};
struct DotList {
  int32_t* d_ptr = nullptr;    // runs of term k: ptr[k] .. ptr[k+1] - 1
  DotRun* d_runs = nullptr;
  double* d_partial = nullptr;
  int64_t n_items = 0;
};

// skip: optional device flag; when *skip != 0 the launch does nothing
void launch_seg_gemm_f64(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                         int accumulate, double* dot_out, const int32_t* skip, cudaStream_t st);
// tiles of mode TM_STORE_DOTS (product and per-segment dots in one pass)
void launch_seg_gemm_f64_dots(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                              int accumulate, double* dot_out, const int32_t* skip, cudaStream_t st);
// the same task lists in double-float arithmetic (matvec_df.cu): the input,
// the operators and the intermediates hold float32 pairs (hi, lo) in their
// 8-byte slots, the output is float64
void launch_seg_gemm_df(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                        int accumulate, cudaStream_t st);
void launch_seg_gemm_df_dots(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                             int accumulate, double* dot_out, cudaStream_t st);
// dst[i] = the double-float pair of src[i] (n elements)
void launch_split_pairs(const double* src, double* dst, int64_t n, cudaStream_t st);

// ------------------------------------------------------------ host pair info
struct PairH {
  int32_t term, s_out, s_in, flags;
  int64_t a_off, b_off;  // element offsets in the FP64 operator arena (ld = cols)
  int32_t order;         // two-GEMM pairs: 0 = (A Psi) B^T first A, 1 = A (Psi B^T)
};

}  // namespace dmrg

// ------------------------------------------------------------ the superblock
struct dmrg_sb {
  int32_t S = 0, n_terms = 0, batch = 0;
  std::vector<int32_t> r, c;
  std::vector<int64_t> off;  // [S+1]
  int64_t D = 0;
  std::vector<double> coeffs;  // host [batch][n_terms]
  bool coeffs_set = true;      // false from the start of a dmrg_set_coeffs until it has gone through
  double* d_coeffs = nullptr;  // device [batch][n_terms]
  double* h_coeffs_pinned = nullptr;  // pinned staging copy of coeffs for dmrg_set_coeffs
  std::vector<dmrg::PairH> pairs;
  double* d_ops = nullptr;     // FP64 operator arena
  char* df_mem = nullptr;      // tiles, dot partials, d_ops_df and d_x_df of the double-float products (at the first)
  double* d_ops_df = nullptr;  // the same arena as double-float pairs (first double-float product)
  double* d_x_df = nullptr;    // [batch][D] the double-float product's input as pairs
  int64_t ops_elems = 0;
  double flops = 0;            // algorithmic flops of one product, one member

  // FP64 task lists
  dmrg::TaskListF64 f64_fwd1, f64_fwd2;   // forward: intermediates, outputs
  dmrg::TaskListF64 f64_bwd1, f64_bwd2;   // H^T g
  dmrg::TaskListF64 f64_dot1, f64_dot2;   // per-pair <g, A psi B^T>
  dmrg::TaskListF64 f64_pdot2;            // H psi and per-term <psi, (A_k x B_k) psi> in one pass (after f64_dot1)
  dmrg::DotList dot, pdot, pdot_df;       // term sums of f64_dot2, of f64_pdot2, of its double-float tiles
  double* d_T = nullptr;                  // FP64 intermediate workspace
  int64_t T_elems = 0;
  int64_t T_fwd_elems = 0;               // the part of it the forward product uses
  double* d_scratch = nullptr;  // small reduction scratch (batch norms)
  double* d_red = nullptr;      // [batch][chunks] reduction partials outside Lanczos

  // Lanczos state (allocated on first use)
  int32_t lz_cap = 0;  // Krylov capacity (max_iter + 1)
  double* lz_V = nullptr;        // [lz_cap][batch][D]
  double* lz_w = nullptr;        // [batch][D]
  double* lz_vcur = nullptr;     // [batch][D]
  double* lz_partial = nullptr;  // [batch][nchunk][lz_cap]
  double* lz_h = nullptr;        // Gram-Schmidt coefficients of passes A, B, C: [3][batch][lz_cap]
  double* lz_npart = nullptr;    // |w|^2 chunk partials after passes A, B, C: [3][batch][nchunk]
  int32_t* lz_gate = nullptr;    // [batch] 1: run the second full pass (C); then [batch] block counts
  double* lz_ab = nullptr;       // alpha [batch][lz_cap], beta [batch][lz_cap]
  double* lz_s = nullptr;        // Ritz vector [batch][lz_cap]
  double* lz_out = nullptr;      // per member: theta, resid
  int32_t* lz_ctl = nullptr;     // device control words
  int32_t* h_ctl = nullptr;      // host mirror
  int32_t lz_nchunk = 0;
  // float64 refinement (Newton step with mixed CG) buffers, allocated with Lanczos
  float* rf_res = nullptr;       // [batch][D] inner CG vectors (float32)
  float* rf_p = nullptr;
  double* rf_q = nullptr;        // [batch][D] mixed product H p (float64 output)
  float* rf_hp = nullptr;        // (H - theta) p
  float* rf_t = nullptr;
  float* rf_psi32 = nullptr;     // the iterate, rounded for the inner solve
  double* rf_sc = nullptr;       // [batch][8] scalars, then eps
  int32_t* rf_ctl = nullptr;     // [2 batch + 2]
  double* rf_diag = nullptr;     // [batch][D] diag(H) per member (preconditioner)
  float* rf_minv = nullptr;      // [batch][D] 1 / max(diag - theta, delta)
  double* rf_part = nullptr;     // [4][batch][nchunk] reduction partials
  // terms with diagonal blocks (s_out == s_in): their diagonals, [n][D]
  std::vector<int32_t> dg_terms;
  int32_t* d_dg_terms = nullptr;
  double* d_dg = nullptr;
  void* lz_graphs[8] = {};       // cached cudaGraphExec_t per (prec, K) slot
  int32_t lz_graph_key[8] = {};
  // the allocations that hold the small arrays of the superblock and of its solver buffers
  char *slab = nullptr, *lz_slab = nullptr;
  size_t slab_bytes = 0, lz_slab_bytes = 0;

  void* tc = nullptr;            // tensor-core path state (matvec_tc.cu)
  int32_t* d_tc_err = nullptr;   // set by a tensor-core kernel whose bounded wait gave up
  int32_t test_stall = 0;        // testing hook: the next tensor-core product issues no copies
  int32_t test_fail_panels = 0;  // testing hook: the next build of tensor-core panels reports out of memory
  int32_t test_force_pending = 0;  // testing hook: the next Lanczos solve's float32 test passes at its first check
  std::vector<double> h_ops;     // host copy of the float64 arena during creation only

  std::string err;
};

namespace dmrg {
// forget the captured Lanczos and CG iterations (the memory they name is about to be replaced)
void lz_drop_graphs(dmrg_sb* sb);
}  // namespace dmrg
