// Grouped sector GEMM in double-float arithmetic: the float64 product's task
// lists (same tiles, segments and outputs as matvec_f64.cu), with every
// multiply-add done on float32 pairs.
//
// A double-float number is an unevaluated pair hi + lo of float32 values
// (about 48 significant bits).  Inputs are float64; each is split into
// hi = RN24(v) and lo = RN24(v - hi) with integer instructions, products use
// Dekker's splitting-free form with a fused multiply-add (the error of
// hi_a * hi_b is exact, the cross terms are added to it, lo_a * lo_b -- 2^-46
// relative -- is dropped), and sums use Knuth's two-sum, so one multiply-add
// costs 12 float32 operations and has a relative error near 2^-46; the pair
// is renormalised after every K tile of 16 (without it the low sum's own
// rounding grows like K 2^-48: 1e-12 at K = 200).  GB300
// runs float64 at 1/64 of its float32 rate (2 DFMA per clock per SM against
// 128 FFMA), so the arithmetic alone allows five times the float64 kernel's
// rate; the superblock product runs two to three times as fast as the float64
// kernel, at an accuracy enough for residuals r = H psi - theta psi down to
// |r| ~ 1e-12 |H psi|.  Outputs are written as float64 (hi + lo).  Paper Sec. 3.3: the product x += H y, system,
// environment and connection parts, on the fly.
//
// Every operand holds its elements as float32 pairs (hi, lo) in 8-byte slots,
// already split: the operator arena (split once per superblock), the
// wavefunction (split once per product) and the intermediates, which phase 1
// writes as its renormalised (s, c) sums (48 bits, no rounding to float64
// between the two GEMMs).
//
// The two groups of an output's segments are chains of their own, added in
// float64: one chain over both carries the first group's rounding through the
// second (error of a product against float64, relative to |y|: 6.4e-14 with
// one chain, 4.7e-14 with two on a real m = 1000 superblock, 1.3e-14 and 5.6e-15 on
// the 32-site chain at m = 1000; it costs 0.3 to 2 % of the time, 5 % on the
// 2 x 32 ladder at m = 400).
//
// Bound: instruction issue (80 % of the slots on wide sectors, 66-73 % on the
// ladder).  Measured against 64 x 64 tiles of 256 threads: the 32-site chain
// at m = 1000 472 -> 277 us, 16 sectors 16..512 wide 4.96 -> 4.23 ms, the 2 x 32
// ladder at m = 1000 (16 members) 3.15 -> 2.90 ms, with the per-term dots 4.21
// -> 3.62 ms; a real m = 1000 superblock (blocks up to 424 wide, 16 members) 37.9
// -> 37.0 ms (24 x 24 tiles; 40.2 with 16 x 16), with the dots 41.3 -> 40.5 ms (16 x
// 16: the dots need a third set of sums).  Tiles of 32 x 32 (16 sums a thread)
// were slower: 6.4 ms on the 16 sectors, too few warps for their registers.

#include <algorithm>

#include "df.cuh"
#include "internal.h"
#include "seg_tile.cuh"

namespace dmrg {

// the 8 bytes of a pair slot as (hi, lo): hi is the low word (float2 layout)
__device__ __forceinline__ float2 df_bits(double v) {
  return make_float2(__int_as_float(__double2loint(v)), __int_as_float(__double2hiint(v)));
}
__device__ __forceinline__ double df_slot(float s, float c) {  // (s, c) renormalised into one slot
  const float hi = __fadd_rn(s, c);
  const float lo = __fsub_rn(c, __fsub_rn(hi, s));
  return __hiloint2double(__float_as_int(lo), __float_as_int(hi));
}

struct ArDF {
  using Acc = float2;   // double-float sum (s, c)
  using Coef = float2;
  using Dot = double;
  static constexpr bool unrolled_tail = false;
  static __device__ __forceinline__ float2 zero() { return make_float2(0.0f, 0.0f); }
  static __device__ __forceinline__ void fma(double a, double b, float2& c) { df_fma(df_bits(a), df_bits(b), c.x, c.y); }
  // renormalise (fast two-sum, |c| << |s|): c restarts near ulp(s) / 2, so
  // its own rounding stays near 2^-48 |s| per K step of the next chunk
  static __device__ __forceinline__ void end_chunk(float2& a) {
    const float t = __fadd_rn(a.x, a.y);
    a.y = __fsub_rn(a.y, __fsub_rn(t, a.x));
    a.x = t;
  }
  static __device__ __forceinline__ float2 coef(double c) { return df_split(c); }
  static __device__ __forceinline__ double scaled(double v, float2 c) {
    const float2 p = df_mul(df_bits(v), c);
    return __hiloint2double(__float_as_int(p.y), __float_as_int(p.x));
  }
  static __device__ __forceinline__ double value(float2 a) { return df_value(a.x, a.y); }
  static __device__ __forceinline__ double slot(float2 a) { return df_slot(a.x, a.y); }
  // dots with the wavefunction's pairs, in float64
  static __device__ __forceinline__ double dot_zero() { return 0.0; }
  static __device__ __forceinline__ void dot(float2 a, double x, double& p) {
    const float2 v = df_bits(x);
    p = ::fma(df_value(a.x, a.y), df_value(v.x, v.y), p);
  }
  static __device__ __forceinline__ double dot_warp(double p) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    return p;
  }
};


// BMAX: the widest tile edge of the list
template <bool DOTS, int BMAX>
__global__ void __launch_bounds__(SEG_THREADS, 8)
seg_gemm_df_kernel(const TileF64* __restrict__ tiles, const SegF64* __restrict__ segs, Bufs bufs,
                   const double* __restrict__ coef, int n_terms, int batch, int accumulate,
                   double* __restrict__ dot_out) {
  __shared__ SegSmem<BMAX> sm;
  const TileF64 t = tiles[blockIdx.x / batch];
  const int member = blockIdx.x % batch;
#define DF_CASE(I, J)                                                                                       \
  case (I) | ((J) << 8):                                                                                    \
    if constexpr (8 * I <= BMAX && 8 * J <= BMAX) seg_tile<ArDF, I, J, DOTS>(t, member, batch, segs, bufs, coef, n_terms, accumulate, dot_out, sm); \
    break;
  switch (t.shape) {
    SEG_SHAPES(DF_CASE)
    default: break;  // the host builds only these shapes
  }
#undef DF_CASE
}

void launch_seg_gemm_df(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                        int accumulate, cudaStream_t st) {
  if (tl.n_tiles_df == 0) return;
  (tl.wide_df ? seg_gemm_df_kernel<false, SEG_BWIDE> : seg_gemm_df_kernel<false, 16>)
      <<<(unsigned)(tl.n_tiles_df * batch), SEG_THREADS, 0, st>>>(tl.d_tiles_df, tl.d_segs, bufs, coef, n_terms, batch,
                                                                 accumulate, nullptr);
}

void launch_seg_gemm_df_dots(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                             int accumulate, double* dot_out, cudaStream_t st) {
  if (tl.n_tiles_df == 0) return;
  seg_gemm_df_kernel<true, 16><<<(unsigned)(tl.n_tiles_df * batch), SEG_THREADS, 0, st>>>(
      tl.d_tiles_df, tl.d_segs, bufs, coef, n_terms, batch, accumulate, dot_out);
}

// dst[i] = the pair (hi, lo) of src[i] in its 8-byte slot
__global__ void k_split_pairs(const double* __restrict__ src, double* __restrict__ dst, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float2 p = df_split(src[i]);
    dst[i] = __hiloint2double(__float_as_int(p.y), __float_as_int(p.x));
  }
}

void launch_split_pairs(const double* src, double* dst, int64_t n, cudaStream_t st) {
  if (n <= 0) return;
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4096);  // grid-stride beyond
  k_split_pairs<<<(unsigned)blocks, 256, 0, st>>>(src, dst, n);
}

}  // namespace dmrg
