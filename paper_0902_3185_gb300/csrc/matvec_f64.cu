// Grouped FP64 sector GEMM: every (term, sector pair) product of the
// superblock Hamiltonian in one launch per phase, on the CUDA cores in
// float64.
//
// Paper Sec. 3.3: the product x += H y is done per symmetry block, on the
// fly, as system, environment and connection parts.  Here each output tile
// of a block Y_s (or of an intermediate A Psi / Psi B^T) walks over a list of
// segments, each a plain product L (M x K) * R (K x N) with its own layout
// and coefficient, and accumulates them in registers (seg_tile.cuh).  One
// tile writes each output element exactly once, so results do not depend on
// scheduling.
//
// Measured against 64 x 64 tiles of 256 threads with one chunk in flight and
// the two output groups in launches of their own: one product of the 12-site
// ladder at m = 60 (2 members) 145 -> 26 us, of the 32-site chain at m = 200
// 107 -> 27 us, at m = 1000 1428 -> 742 us, of the 2 x 32 ladder at m = 400 (4
// members) 708 -> 212 us, at m = 1000 (16 members) 7.80 -> 7.43 ms, of 16 sectors
// 16..512 wide 17.3 -> 14.0 ms (1.15 TFLOP/s; the float64 unit is 95-97 % busy), of
// a real m = 1000 superblock (16 members) 135.0 -> 131.6 ms.

#include "internal.h"
#include "seg_tile.cuh"

namespace dmrg {

struct ArF64 {
  using Acc = double;
  // a coefficient: 1 and -1, the usual ones, cost no float64 instruction (nor
  // does telling them: a float64 compare runs on the same unit)
  struct Coef {
    double c;
    uint32_t sign;
    bool unit;
  };
  using Dot = double;
  static constexpr bool unrolled_tail = true;
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ void fma(double a, double b, double& c) { c = ::fma(a, b, c); }
  static __device__ __forceinline__ void end_chunk(double&) {}
  static __device__ __forceinline__ Coef coef(double c) {
    const uint32_t hi = (uint32_t)__double2hiint(c);
    return Coef{c, hi & 0x80000000u, (hi & 0x7fffffffu) == 0x3ff00000u && __double2loint(c) == 0};
  }
  static __device__ __forceinline__ double scaled(double v, const Coef& f) {
    if (f.unit) return __hiloint2double((int)((uint32_t)__double2hiint(v) ^ f.sign), __double2loint(v));
    return v * f.c;
  }
  static __device__ __forceinline__ double value(double a) { return a; }
  static __device__ __forceinline__ double slot(double a) { return a; }
  static __device__ __forceinline__ double dot_zero() { return 0.0; }
  static __device__ __forceinline__ void dot(double a, double x, double& p) { p = ::fma(a, x, p); }
  static __device__ __forceinline__ double dot_warp(double p) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    return p;
  }
};


// BMAX: the widest tile edge of the list
template <bool DOTS, int BMAX>
__global__ void __launch_bounds__(SEG_THREADS, 8)
seg_gemm_f64_kernel(const TileF64* __restrict__ tiles, const SegF64* __restrict__ segs, Bufs bufs,
                    const double* __restrict__ coef, int n_terms, int batch, int accumulate,
                    double* __restrict__ dot_out, const int32_t* __restrict__ skip) {
  __shared__ SegSmem<BMAX> sm;
  if (skip && *skip) return;
  const TileF64 t = tiles[blockIdx.x / batch];
  const int member = blockIdx.x % batch;
#define F64_CASE(I, J)                                                                                       \
  case (I) | ((J) << 8):                                                                                     \
    if constexpr (8 * I <= BMAX && 8 * J <= BMAX) seg_tile<ArF64, I, J, DOTS>(t, member, batch, segs, bufs, coef, n_terms, accumulate, dot_out, sm); \
    break;
  switch (t.shape) {
    SEG_SHAPES(F64_CASE)
    default: break;  // the host builds only the shapes above
  }
#undef F64_CASE
}

void launch_seg_gemm_f64_dots(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                              int accumulate, double* dot_out, const int32_t* skip, cudaStream_t st) {
  if (tl.n_tiles == 0) return;
  seg_gemm_f64_kernel<true, 16><<<(unsigned)(tl.n_tiles * batch), SEG_THREADS, 0, st>>>(
      tl.d_tiles, tl.d_segs, bufs, coef, n_terms, batch, accumulate, dot_out, skip);
}

void launch_seg_gemm_f64(const TaskListF64& tl, const Bufs& bufs, const double* coef, int n_terms, int batch,
                         int accumulate, double* dot_out, const int32_t* skip, cudaStream_t st) {
  if (tl.n_tiles == 0) return;
  (tl.wide ? seg_gemm_f64_kernel<false, SEG_BWIDE> : seg_gemm_f64_kernel<false, 16>)
      <<<(unsigned)(tl.n_tiles * batch), SEG_THREADS, 0, st>>>(tl.d_tiles, tl.d_segs, bufs, coef, n_terms, batch,
                                                              accumulate, dot_out, skip);
}

}  // namespace dmrg
