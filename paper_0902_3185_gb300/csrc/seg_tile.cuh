// The grouped sector product on the CUDA cores, shared by the float64 and the
// double-float arithmetic: one thread block per output tile of one batch
// member, walking over a list of segments L (M x K) * R (K x N).
//
// What bounds it.  GB300 issues 2 float64 fused multiply-adds per clock per SM
// (one unit shared by the SM's four schedulers: a warp's instruction takes 16
// cycles of it), so the product is bound by that unit as soon as a few warps
// per SM have work, and by the length of one output element's chain of
// multiply-adds when an SM has too little of it.  Hence small tiles: 8, 16 or,
// in lists that fill the chip several times over, 24 outputs a side, 64 threads,
// at most nine chains per thread.  Operand traffic does not matter at this rate
// (a 16 x 16 tile reads 1 byte per multiply-add from L2), padding and idle SMs
// do: sector blocks are 1..80 wide in a DMRG superblock, up to 512 in the
// widest, and a tile is padded to multiples of 8 only.  Every SM holds many
// such blocks, which hides the latency of each one's loads and barriers.
//
// The segments of a tile are one flat sequence of K chunks of 16, copied by
// cp.async (8 bytes per element, zero outside the operands) into a ring of
// four shared-memory stages, three chunks ahead of the multiply-adds and
// across segment boundaries; one barrier per chunk.  A segment's coefficient
// scales one operand: each thread scales the elements it copied itself, after
// its own copies have landed and before the barrier that publishes them.
//
// Every output element is one chain per group of segments, over the group's
// segments in list order and over k in increasing order, and the two chains'
// values are added in float64, whatever the tile shape, the same chains on
// every call.
#pragma once

#include <cstdint>

#include "internal.h"

namespace dmrg {

// tile shapes 8 I x 8 J (a kernel for lists up to BMAX wide compiles those that fit)
#define SEG_SHAPES(CASE) \
  CASE(1, 1) CASE(1, 2) CASE(2, 1) CASE(2, 2) CASE(1, 3) CASE(2, 3) CASE(3, 1) CASE(3, 2) CASE(3, 3)
constexpr int SEG_BWIDE = 24;  // widest tile edge of a wide list

constexpr int SEG_THREADS = 64;
constexpr int SEG_BK = 16;      // K chunk
constexpr int SEG_STAGES = 4;   // ring of chunks
constexpr int SEG_SMEM_SEGS = 32;  // segments prepared in shared memory (later ones when they are reached)

// A segment as one tile of one member sees it: the operands at the tile's first
// row and column, the coefficient.  The first SEG_SMEM_SEGS of a tile are
// prepared by its threads side by side, so that neither the copies nor the
// multiply-adds wait for a descriptor or a coefficient between segments: a
// product of the 12-site ladder at m = 60 27.6 -> 25.6 us, the per-term dots of
// the m = 1000 ladder 3.69 -> 3.62 ms.
struct SegView {
  const double *L, *R;
  double cf;
  int32_t ldl, ldr, K;
  int8_t l_trans, r_trans, scale, pad;
};

template <int BMAX>  // widest tile edge
struct SegSmem {
  double L[SEG_STAGES][SEG_BK][BMAX + 1];  // 8-byte slots: float64 values or float32 pairs
  double R[SEG_STAGES][SEG_BK][BMAX + 1];
  SegView segs[SEG_SMEM_SEGS];
  double* base[NBUF];  // the launch's buffers
};

__device__ __forceinline__ void cp_async8(double* dst, const double* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int n = valid ? 8 : 0;  // 0: the 8 bytes are zero-filled and src is not read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ SegView seg_view(const SegF64& s, const TileF64& t, int member, double* const* base,
                                            const double* __restrict__ coef, int n_terms) {
  SegView v;
  v.L = base[s.l_buf] + s.l_off + (int64_t)member * s.l_bs + (s.l_trans ? (int64_t)t.m0 : (int64_t)t.m0 * s.ldl);
  v.R = base[s.r_buf] + s.r_off + (int64_t)member * s.r_bs + (s.r_trans ? (int64_t)t.n0 * s.ldr : (int64_t)t.n0);
  v.cf = coef[(int64_t)member * n_terms + s.term];
  v.ldl = s.ldl;
  v.ldr = s.ldr;
  v.K = s.K;
  v.l_trans = (int8_t)s.l_trans;
  v.r_trans = (int8_t)s.r_trans;
  v.scale = (int8_t)s.scale;
  v.pad = 0;
  return v;
}

// Copies one chunk after the other of a tile's segments into the ring.
template <int BM, int BN, class SMEM>
struct SegCopier {
  static constexpr int SL = BM * SEG_BK / SEG_THREADS, SR = BN * SEG_BK / SEG_THREADS;
  const TileF64& t;
  const SegF64* __restrict__ segs;
  const double* __restrict__ coef;
  SMEM& sm;
  const int n_terms, member, tid;
  int q, k0 = 0, K = 0, l_trans = 0, r_trans = 0;
  const double *lp = nullptr, *rp = nullptr;  // this thread's first slot
  int32_t ldl = 0, ldr = 0;

  __device__ __forceinline__ SegCopier(const TileF64& t_, const SegF64* segs_, const double* coef_, int n_terms_,
                                       SMEM& sm_, int member_)
      : t(t_), segs(segs_), coef(coef_), sm(sm_), n_terms(n_terms_), member(member_), tid(threadIdx.x), q(t_.seg_begin) {
    open();
  }
  __device__ __forceinline__ SegView seg(int i) const {
    const int l = i - t.seg_begin;
    return l < SEG_SMEM_SEGS ? sm.segs[l] : seg_view(segs[i], t, member, sm.base, coef, n_terms);
  }
  // Element slot e of thread tid in an operand with an outer index o of width B
  // (rows of L, columns of R) and the K index: consecutive threads run along
  // the contiguous direction, K (k_fast) or o.  `step` is the slot's distance
  // from the thread's slot 0 as o and k.
  template <int B>
  static __device__ __forceinline__ void slot(int tid, int e, bool k_fast, int& o, int& k) {
    if (k_fast) {
      o = (tid + e * SEG_THREADS) / SEG_BK;
      k = (tid + e * SEG_THREADS) % SEG_BK;
    } else if (SEG_THREADS % B == 0) {
      k = (tid + e * SEG_THREADS) / B;
      o = (tid + e * SEG_THREADS) % B;
    } else {  // runs of 8 along o
      k = tid / 8 + 8 * (e / (B / 8));
      o = tid % 8 + 8 * (e % (B / 8));
    }
  }
  template <int B>
  static __device__ __forceinline__ int64_t step(int e, bool k_fast, int32_t ld) {
    if (k_fast) return (int64_t)ld * (e * SEG_THREADS / SEG_BK);
    if (SEG_THREADS % B == 0) return (int64_t)ld * (e * SEG_THREADS / B);
    return (int64_t)ld * (8 * (e / (B / 8))) + 8 * (e % (B / 8));
  }
  static __device__ __forceinline__ void l_slot(int tid, int e, int trans, int& m, int& k) {
    slot<BM>(tid, e, !trans, m, k);
  }
  static __device__ __forceinline__ void r_slot(int tid, int e, int trans, int& n, int& k) {
    slot<BN>(tid, e, trans, n, k);
  }
  __device__ __forceinline__ void open() {
    if (q >= t.seg_end) return;
    const SegView s = seg(q);
    k0 = 0;
    K = s.K;
    l_trans = s.l_trans;
    r_trans = s.r_trans;
    ldl = s.ldl;
    ldr = s.ldr;
    int m, n, kl, kr;
    l_slot(tid, 0, l_trans, m, kl);
    r_slot(tid, 0, r_trans, n, kr);
    lp = s.L + (l_trans ? (int64_t)kl * ldl + m : (int64_t)m * ldl + kl);
    rp = s.R + (r_trans ? (int64_t)n * ldr + kr : (int64_t)kr * ldr + n);
  }
  // the next chunk into a stage (an empty group past the last one)
  __device__ __forceinline__ void copy(int stage) {
    if (q < t.seg_end) {
      const double* none = sm.base[BUF_OPS];
#pragma unroll
      for (int e = 0; e < SL; ++e) {
        int m, k;
        l_slot(tid, e, l_trans, m, k);
        const bool in = t.m0 + m < t.M && k0 + k < K;
        cp_async8(&sm.L[stage][k][m], in ? lp + step<BM>(e, !l_trans, ldl) : none, in);
      }
#pragma unroll
      for (int e = 0; e < SR; ++e) {
        int n, k;
        r_slot(tid, e, r_trans, n, k);
        const bool in = t.n0 + n < t.N && k0 + k < K;
        cp_async8(&sm.R[stage][k][n], in ? rp + step<BN>(e, r_trans, ldr) : none, in);
      }
      lp += l_trans ? (int64_t)SEG_BK * ldl : SEG_BK;
      rp += r_trans ? SEG_BK : (int64_t)SEG_BK * ldr;
      k0 += SEG_BK;
      if (k0 >= K) {
        ++q;
        open();
      }
    }
    cp_async_commit();
  }
};

// One output tile.  AR is the arithmetic: its sums (Acc), a multiply-add, the
// scaling of a slot, the end of a chunk and the value of a sum.  Thread (ty,
// tx) = (tid / 8, tid % 8) holds outputs (ty + 8 i, tx + 8 j).
template <class AR, int NI, int NJ, bool DOTS, class SMEM>
__device__ __forceinline__ void seg_tile(const TileF64& t, int member, int batch, const SegF64* __restrict__ segs,
                                         const Bufs& bufs, const double* __restrict__ coef, int n_terms,
                                         int accumulate, double* __restrict__ dot_out, SMEM& sm) {
  constexpr int BM = 8 * NI, BN = 8 * NJ;
  using Acc = typename AR::Acc;
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, lane = tid & 31, wid = tid >> 5;
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NBUF; ++i) sm.base[i] = bufs.p[i];
  }
  __syncthreads();
  const int ns = min(t.seg_end - t.seg_begin, SEG_SMEM_SEGS);
  for (int i = tid; i < ns; i += SEG_THREADS)
    sm.segs[i] = seg_view(segs[t.seg_begin + i], t, member, sm.base, coef, n_terms);
  __syncthreads();
  SegCopier<BM, BN, SMEM> cp(t, segs, coef, n_terms, sm, member);
  constexpr bool TWO = !DOTS;  // the two groups' sums kept apart (held: the first group's value)
  Acc acc[NI][NJ];
  double held[TWO ? NI : 1][TWO ? NJ : 1];
  double sum[DOTS ? NI : 1][DOTS ? NJ : 1];
#pragma unroll
  for (int i = 0; i < NI; ++i)
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      acc[i][j] = AR::zero();
      if (TWO) held[TWO ? i : 0][TWO ? j : 0] = 0.0;
      if (DOTS) sum[DOTS ? i : 0][DOTS ? j : 0] = 0.0;
    }
  // the output block of this member; (m, n) at m * ldc + n
  const int64_t c0 = t.c_off + (int64_t)member * t.c_bs;
  // DOTS: the wavefunction at this thread's outputs, 0 outside
  double xo[DOTS ? NI : 1][DOTS ? NJ : 1];
  if (DOTS) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int m = t.m0 + ty + 8 * i, n = t.n0 + tx + 8 * j;
        xo[DOTS ? i : 0][DOTS ? j : 0] =
            m < t.M && n < t.N ? bufs.p[BUF_X][c0 + (int64_t)m * t.ldc + n] : 0.0;
      }
  }
#pragma unroll
  for (int c = 0; c < SEG_STAGES - 1; ++c) cp.copy(c);
  int stage = 0;
  for (int q = t.seg_begin; q < t.seg_end; ++q) {
    const SegView s = cp.seg(q);
    const int K = s.K, scale = s.scale;
    const int lt = s.l_trans, rt = s.r_trans;
    if (TWO && q == t.seg_mid && q > t.seg_begin) {  // the second group's sums start from zero
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          held[TWO ? i : 0][TWO ? j : 0] = AR::value(acc[i][j]);
          acc[i][j] = AR::zero();
        }
    }
    const double cf = s.cf;
    const typename AR::Coef f = AR::coef(cf);
    for (int k0 = 0; k0 < K; k0 += SEG_BK) {
      cp_async_wait<SEG_STAGES - 2>();
      if (scale == 1) {
#pragma unroll
        for (int e = 0; e < cp.SL; ++e) {
          int m, k;
          cp.l_slot(tid, e, lt, m, k);
          sm.L[stage][k][m] = AR::scaled(sm.L[stage][k][m], f);
        }
      } else if (scale == 2) {
#pragma unroll
        for (int e = 0; e < cp.SR; ++e) {
          int n, k;
          cp.r_slot(tid, e, rt, n, k);
          sm.R[stage][k][n] = AR::scaled(sm.R[stage][k][n], f);
        }
      }
      __syncthreads();  // this chunk is published, and every thread is done with the previous one
      cp.copy((stage + SEG_STAGES - 1) % SEG_STAGES);
      const int kmax = min(SEG_BK, K - k0);
      auto step = [&](int k) {
        double a[NI], b[NJ];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = sm.L[stage][k][ty + 8 * i];
#pragma unroll
        for (int j = 0; j < NJ; ++j) b[j] = sm.R[stage][k][tx + 8 * j];
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
          for (int j = 0; j < NJ; ++j) AR::fma(a[i], b[j], acc[i][j]);
      };
      // no multiply-adds on the padding of K; float64 takes the remainder by
      // its bits, unrolled, so that the shared-memory loads run ahead of the
      // chains (the double-float loop would outgrow the instruction cache)
      if (kmax == SEG_BK) {
        if (!AR::unrolled_tail && NI * NJ > 4) {
          // two steps at a time: unrolled, the 24-wide double-float chunk is 30 KB
          // of instructions, and the blocks of an SM, each at another place, fetch
          // them from L2 (real m = 1000 superblock, unrolled by 2 / 4 / 8 / 16: 37.0 /
          // 37.1 / 40.6 / 40.8 ms; 64 sectors 16..512 wide 14.1 / 15.1 / 19.5 / 19.6 ms)
#pragma unroll 2
          for (int k = 0; k < SEG_BK; ++k) step(k);
        } else {
#pragma unroll
          for (int k = 0; k < SEG_BK; ++k) step(k);
        }
      } else if (!AR::unrolled_tail) {
        for (int k = 0; k < kmax; ++k) step(k);
      } else {
        int k = 0;
        if (kmax & 8) {
#pragma unroll
          for (int u = 0; u < 8; ++u) step(u);
          k = 8;
        }
        if (kmax & 4) {
#pragma unroll
          for (int u = 0; u < 4; ++u) step(k + u);
          k += 4;
        }
        if (kmax & 2) {
          step(k);
          step(k + 1);
          k += 2;
        }
        if (kmax & 1) step(k);
      }
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) AR::end_chunk(acc[i][j]);
      stage = (stage + 1) % SEG_STAGES;
    }
    if (DOTS) {  // this segment's dot with the wavefunction, then its coefficient
      typename AR::Dot part = AR::dot_zero();
#pragma unroll
      for (int i = 0; i < NI; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          AR::dot(acc[i][j], xo[DOTS ? i : 0][DOTS ? j : 0], part);
          double& v = sum[DOTS ? i : 0][DOTS ? j : 0];
          v = ::fma(cf, AR::value(acc[i][j]), v);
          acc[i][j] = AR::zero();
        }
      const double tot = AR::dot_warp(part);
      if (lane == 0)
        dot_out[((int64_t)(t.dot_base + q - t.seg_begin) * batch + member) * (SEG_THREADS / 32) + wid] = tot;
    }
  }

  double* C = sm.base[t.c_buf] + c0;
  const bool first = t.seg_mid > t.seg_begin || t.seg_end == t.seg_begin, second = t.seg_end > t.seg_mid;
  if (t.mode == TM_DOT) {  // sum over the tile of acc .* C, one partial per warp
    double part = 0.0;
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int m = t.m0 + ty + 8 * i, n = t.n0 + tx + 8 * j;
        if (m < t.M && n < t.N) part = ::fma(AR::value(acc[i][j]), C[(int64_t)m * t.ldc + n], part);
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if (lane == 0) dot_out[(int64_t)blockIdx.x * (SEG_THREADS / 32) + wid] = part;
    return;
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int m = t.m0 + ty + 8 * i;
    if (m >= t.M) continue;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
      const int n = t.n0 + tx + 8 * j;
      if (n >= t.N) continue;
      double* p = C + (int64_t)m * t.ldc + n;
      if (t.c_buf == BUF_T) {  // intermediates stay in the arithmetic's own storage
        *p = AR::slot(acc[i][j]);
        continue;
      }
      if (DOTS) {
        const double v = sum[DOTS ? i : 0][DOTS ? j : 0];
        *p = accumulate ? *p + v : v;
        continue;
      }
      // the first group's sum, then the second's (each a chain of its own)
      const bool both = TWO && first && second;
      const double v1 = both ? held[TWO ? i : 0][TWO ? j : 0] : AR::value(acc[i][j]);
      double y = accumulate ? *p + v1 : v1;
      if (both) y += AR::value(acc[i][j]);
      *p = y;
    }
  }
}

}  // namespace dmrg
