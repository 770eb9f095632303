// Tile lists of the CUDA-core products made on the device, and the sums of
// their per-term dot partials.
#pragma once

#include "internal.h"

namespace dmrg {

// The tiles of up to MAX lists in one launch: output i of a list (its
// descriptor at the origin) becomes tiles first[i] .. first[i+1] - 1, row by
// row of tiles.  Expanding on the device keeps the host from writing and
// copying 80 bytes for each of the tens of thousands of tiles of a superblock,
// which a DMRG step uses once: first double-float product of the 2 x 32 ladder
// at m = 1000 5.2 -> 3.3 ms (the product itself 3.2), of the 32-site chain at m = 1000
// 0.92 -> 0.44 ms (0.30), creation of the ladder's superblock 26.8 -> 25.0 ms.
struct ExpandArgs {
  static constexpr int MAX = 8;
  const TileF64* outs[MAX];
  const int32_t* first[MAX];
  TileF64* tiles[MAX];
  int32_t begin[MAX + 1];  // blocks of list l: begin[l] .. begin[l+1] - 1, one per output
  int n = 0;
  void add(const TileF64* o, const int32_t* f, TileF64* t, int32_t n_outs) {
    outs[n] = o;
    first[n] = f;
    tiles[n] = t;
    if (n == 0) begin[0] = 0;
    begin[n + 1] = begin[n] + n_outs;
    ++n;
  }
};
void launch_expand_tiles(const ExpandArgs& a, cudaStream_t st);

// out[b * n_terms + k] = the sum of term k's partials of member b, in list order
void launch_reduce_terms(const DotList& l, double* out, int batch, int n_terms, cudaStream_t st);

}  // namespace dmrg
