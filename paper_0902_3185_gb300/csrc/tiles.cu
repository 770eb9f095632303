// Tile lists expanded on the device and the per-term sums of dot partials
// (tiles.h).  Both are a few microseconds, bound by launch latency.
#include "tiles.h"

namespace dmrg {

__global__ void __launch_bounds__(128) k_expand_tiles(const ExpandArgs a) {
  int l = 0;
  while ((int)blockIdx.x >= a.begin[l + 1]) ++l;
  const int o = (int)blockIdx.x - a.begin[l];
  const TileF64 t = a.outs[l][o];
  const int32_t f = a.first[l][o], n = a.first[l][o + 1] - f;
  const int bm = 8 * (t.shape & 0xff), bn = 8 * (t.shape >> 8);
  const int across = (t.N + bn - 1) / bn;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    TileF64 u = t;
    u.m0 = i / across * bm;
    u.n0 = i % across * bn;
    if (t.mode == TM_STORE_DOTS) u.dot_base += i * (t.seg_end - t.seg_begin);
    a.tiles[l][f + i] = u;
  }
}

void launch_expand_tiles(const ExpandArgs& a, cudaStream_t st) {
  if (a.n == 0 || a.begin[a.n] == 0) return;
  k_expand_tiles<<<(unsigned)a.begin[a.n], 128, 0, st>>>(a);
}

// One block per (member, term): thread-strided sums over the term's partials
// (element e of the list: item e / SEG_DOT_PARTS, its part e % SEG_DOT_PARTS),
// then a fixed-order block reduction (deterministic).  The items of a term come
// as runs, one per output and segment, an item per tile: the host makes a few
// of them instead of an index per partial.  They are read into shared memory
// side by side and searched there (walked through in global memory they had
// cost 8 us of latency on a product with dots of 60 us).
constexpr int RED_THREADS = 256;
__global__ void __launch_bounds__(RED_THREADS)
k_reduce_terms(const double* __restrict__ part, const int32_t* __restrict__ ptr, const DotRun* __restrict__ runs,
               double* __restrict__ out, int batch, int n_terms) {
  __shared__ double red[RED_THREADS / 32];
  __shared__ DotRun rs[RED_THREADS];
  const int b = blockIdx.x / n_terms, k = blockIdx.x % n_terms;
  const int r_end = ptr[k + 1];
  double t = 0.0;
  unsigned e = threadIdx.x;
  for (int r0 = ptr[k]; r0 < r_end; r0 += RED_THREADS) {
    const int nr = min(RED_THREADS, r_end - r0);
    __syncthreads();
    if ((int)threadIdx.x < nr) rs[threadIdx.x] = runs[r0 + threadIdx.x];
    __syncthreads();
    const unsigned stop = (unsigned)rs[nr - 1].end * SEG_DOT_PARTS;
    for (; e < stop; e += RED_THREADS) {
      const int i = (int)(e / SEG_DOT_PARTS);
      int lo = 0, hi = nr - 1;  // the first run that ends beyond item i
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (rs[mid].end > i) hi = mid;
        else lo = mid + 1;
      }
      const int64_t item = rs[lo].item + (int64_t)(i - rs[lo].first) * rs[lo].stride;
      t += part[(item * batch + b) * SEG_DOT_PARTS + e % SEG_DOT_PARTS];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < RED_THREADS / 32; ++w) s += red[w];
    out[blockIdx.x] = s;
  }
}

void launch_reduce_terms(const DotList& l, double* out, int batch, int n_terms, cudaStream_t st) {
  if (batch * n_terms == 0) return;
  k_reduce_terms<<<(unsigned)(batch * n_terms), RED_THREADS, 0, st>>>(l.d_partial, l.d_ptr, l.d_runs, out, batch, n_terms);
}

}  // namespace dmrg
