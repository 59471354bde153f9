// Tiles, K splits and buffer sizes of the sliced FP64 products (k_gemm_oz.cu):
// host arithmetic only, so that it can be checked without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>

namespace lgw {
namespace oz {

constexpr int BM = 128;         // rows of A per tile
constexpr int KB = 64;          // K elements per block: one 128-byte swizzle row
constexpr int CHUNK_KB = 16;    // 1024 terms per exact sum

// Columns of B per tile: as many as fill the chip with up to `splits` K splits
// (an A tile is loaded once per column tile, so wide tiles load less), no
// wider than B.
inline int tile_cols(int m_tiles, int ncols, int splits, int nsm) {
  int nt = ncols >= 64 ? 64 : (ncols >= 32 ? 32 : 16);
  while (nt > 16 && m_tiles * ((ncols + nt - 1) / nt) * splits * 2 <= nsm) nt /= 2;
  return nt;
}

// K splits of A's M rows by ncols columns over nkb K blocks: the count with
// the fewest K blocks in sequence, a CTA's fixed cost (pipeline fill, eight
// sums joined and stored) standing for four of them.
inline int k_splits(int M, int ncols, int nkb, int nsm) {
  const int m_tiles = (M + BM - 1) / BM;
  const int nt = tile_cols(m_tiles, ncols, std::min(64, nkb), nsm);
  const int tiles = m_tiles * ((ncols + nt - 1) / nt);
  int best = 1;
  long long best_cost = 1LL << 60;
  for (int s = 1; s <= std::min(64, nkb); ++s) {
    const int per = (nkb + s - 1) / s, real = (nkb + per - 1) / per;
    const long long waves = ((long long)tiles * real + nsm - 1) / nsm;
    const long long cost = waves * (per + 4 * ((per + CHUNK_KB - 1) / CHUNK_KB));
    if (cost < best_cost) {
      best_cost = cost;
      best = real;
    }
  }
  return best;
}

// Rows of split partials that `rows` columns of B need when they are taken
// `slice` at a time.  The last, shorter slice counts too: fewer columns get
// more splits, often more than their share of the rows.
inline size_t part_rows(int M, int rows, int slice, int nkb, int nsm) {
  const int full = std::min(rows, slice), tail = rows > slice ? rows % slice : 0;
  size_t n = (size_t)k_splits(M, full, nkb, nsm) * full;
  if (tail > 0) n = std::max(n, (size_t)k_splits(M, tail, nkb, nsm) * tail);
  return n;
}

}  // namespace oz
}  // namespace lgw
