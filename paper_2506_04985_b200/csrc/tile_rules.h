// How the matmul launchers cut their work into tiles: host arithmetic on sizes alone, without CUDA, so that it can be
// compiled and looked at without a GPU.
#pragma once

namespace fpt {

// Columns (N) an 8-bit integer tcgen05.mma of a CTA pair may have with 256 rows: multiples of 32 (of one CTA with 128
// rows: of 16).
constexpr bool umma_i8_pair_width(int n) { return n >= 32 && n <= 256 && n % 32 == 0; }

// Tile width of the CTA-pair kernel for packed codes, plain epilogue: tiles are dealt out in rounds of `pairs`, and the
// width with the smallest rounds x width wins; among equal costs the wider (fewer tiles, less activation traffic).  (A
// tile's time falls less than its width, because the converters' chain per k-block does not shrink with the tile: one
// round of 256 / 224 columns of 2048 tokens x 4096 takes 18.2 / 17.2 us, x 14336 41.6 / 40.3.)
constexpr int kPairRows = 256, kPairWidth = 256, kPairNarrow = 224;
static_assert(umma_i8_pair_width(kPairWidth) && umma_i8_pair_width(kPairNarrow), "instruction shape");
inline int pair_tile_width(int M, int N, int pairs) {
  const long long rows = (M + kPairRows - 1) / kPairRows;
  auto cost = [&](int tn) { return (rows * ((N + tn - 1) / tn) + pairs - 1) / pairs * tn; };
  return cost(kPairNarrow) * 100 < cost(kPairWidth) * 98 ? kPairNarrow : kPairWidth;
}

}  // namespace fpt
