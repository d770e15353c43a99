// How the reduction range of K = X X^T is split over the GPU, and the size of the
// partial sums (host arithmetic only).
#pragma once

#include <stddef.h>

#include <algorithm>

namespace dfjk {

// Partial sums are written out while those of all splits take at most this (see
// k_gemm_sliced); DFJK_OZ_SIMPLE=1 writes them always, within the second figure.
constexpr size_t K_PART_BYTES = (size_t)64 << 20, K_PART_BYTES_SIMPLE = (size_t)4 << 30;

struct KShape {
  int nao = 0, tiles = 0;  // tiles: output tiles that meet the lower triangle
  size_t block_bytes = 0;  // operand slices of one K block, all rows
  size_t range_bytes = 0;  // operand slices of one split, about
  bool ordered = true;     // the persistent kernel: splits can add in order, without partial sums
};
struct KSplit {
  int n = 1, per = 1;     // splits, K blocks in each
  bool partials = false;  // n nao^2 doubles of partial sums
};

inline int k_tiles(int nao, int bm, int bn) {
  int tiles = 0;
  for (int i = 0; i * bm < nao; ++i)
    for (int j = 0; j * bn < nao; ++j)
      if (j * bn <= i * bm + bm - 1) ++tiles;
  return tiles;
}

// Splits asked for: ranges of range_bytes, but enough of them for two tiles per SM.
inline int k_want(const KShape &s, int nkb) {
  const int per = (int)std::max<size_t>(1, s.range_bytes / s.block_bytes);
  const size_t n2 = (size_t)s.nao * s.nao * 8;
  const int most = s.ordered ? nkb : (int)std::max<size_t>(1, K_PART_BYTES_SIMPLE / n2);
  const int n = std::min((nkb + per - 1) / per, most);
  return std::max(n, std::min(nkb, (2 * 152 + s.tiles - 1) / s.tiles));
}

inline KSplit k_split(const KShape &s, int nkb) {
  KSplit r;
  r.n = k_want(s, nkb);
  r.per = (nkb + r.n - 1) / r.n;
  r.n = (nkb + r.per - 1) / r.per;  // the rounding makes this jump: at nao = 450, 81 blocks give 14 splits, 80 give 16
  r.partials = !s.ordered || (size_t)r.n * s.nao * s.nao * 8 <= K_PART_BYTES;
  return r;
}

// Doubles of partial sums that hold those of every range of at most nkb_max K blocks: a
// shorter range can have more splits than a longer one and can take partial sums where
// the longer one does not, but k_want grows with the range and bounds its splits.
inline size_t k_part_doubles(const KShape &s, int nkb_max) {
  const size_t n2 = (size_t)s.nao * s.nao, want = (size_t)k_want(s, nkb_max);
  return (s.ordered ? std::min(want, K_PART_BYTES / (n2 * 8)) : want) * n2;
}

}  // namespace dfjk
