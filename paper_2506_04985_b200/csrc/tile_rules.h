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

// How a launch of the kernel for one-byte codes (gemm_wt_pair.cu) cuts its work: tokens of a tile, and whether two CTA
// pairs share one.  The cut with the least time, by what was measured at 1.9 GHz (ns).  Tiles are dealt out in rounds of
// `pairs`; a k-block takes what the hand-overs take up to 96 tokens (160), then more and more the MMAs (274 at 256 tokens);
// a tile with one accumulator 1.2 us more, in which it is emptied.  Where the chip is full the power limit sets the pace
// instead, 95 a k-block and 1.08 a token of it over all pairs.  Start and end of a launch 6500 and 14.5 a token of a tile; a
// shared tile halves the k-blocks for 1.4 us.
// (us, 32 / 64 / .. / 256 tokens: 2048x6144x4096 133 / 75 / 56 / 46 / 44 / 40 / 45 / 40; 777x6144x4096 58 / 36 / 26 / 26 / 22 /
// 23.5 / 26 / 29; 512x4096x14336 81 / 44 / 45 / 32 / 30 / 33 / 37 / 41; 128x4096x14336, shared: 64 tokens 18.8, else 24.8.)
// With rows of fewer than 2048 codes the plain epilogue sets the pace of the rounds but the last, 64 tokens at a time (32 of
// each half): 600, 7 a token and 7 a token of whole steps where there is a second accumulator, else 200, 11.7 and 9, and 0.3
// of the main loop, since both want the same issue slots.
// (8-bit codes, 32 / 64 / .. / 256 tokens: 8192x4096x128 83 / 51 / 47 / 39 / 51 / 48 / 47 / 44; 1500x3072x256 14.6 / 10.8 / 10.0 /
// 9.1 / 11.2 / 11.8 / 13.0 / 8.8, where tiles of 64 were taken when the epilogue was left out.)
constexpr int kWtRows = 256, kWtTokens = 256, kWtStage = 256;        // weight rows, tokens at most; codes of a weight stage
constexpr int kWtDouble = 128;                                       // tokens up to which there are two accumulators
struct WtCut { int tn, ksplit; long long ns; };
inline WtCut wt_cut(int M, int N, int K, int pairs, int quads, bool plain = true) {
  const long long rows = (N + kWtRows - 1) / kWtRows, kblocks = 2 * ((K + kWtStage - 1) / kWtStage);
  constexpr int kBlockNs[kWtTokens / 32] = {160, 160, 168, 176, 183, 203, 240, 274};
  WtCut best = {32, 1, -1};
  for (int tn = kWtTokens; tn >= 32; tn -= 32) {
    const bool twice = tn <= kWtDouble;
    const long long tiles = rows * ((M + tn - 1) / tn), rounds = (tiles + pairs - 1) / pairs;
    const long long block = kBlockNs[tn / 32 - 1], loop = kblocks * block, ends = 6500 + 29 * tn / 2;
    const long long tile = loop + (twice ? 100 : 1200);
    const int steps = (tn + 63) / 64 * 64;
    const long long epilogue = !plain || K >= 2048 ? 0 : (twice ? 600 + 7 * (steps + tn) : 200 + 9 * steps + 117 * tn / 10) + loop * 3 / 10;
    const long long paced = tile + (rounds - 1) * (tile > epilogue ? tile : epilogue);
    const long long power = tiles * kblocks * (9500 + 108 * tn) / (100ll * pairs);
    const long long ns = (paced > power ? paced : power) + ends;
    if (best.ns < 0 || ns < best.ns) best = {tn, 1, ns};
    if (tiles <= quads && kblocks >= 8) {
      const long long ns2 = (kblocks + 3) / 4 * 2 * block + 1400 + ends;
      if (ns2 < best.ns) best = {tn, 2, ns2};
    }
  }
  return best;
}

}  // namespace fpt
