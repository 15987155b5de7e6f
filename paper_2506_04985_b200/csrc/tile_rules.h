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

// Whether the quantiser should leave 4-bit codes one byte each for that kernel, for a linear with the plain epilogue.  Both
// sides measured (us with the quantise pass, packed / one byte) over 3800 shapes; the rule is 0.25 % behind the better side on
// the average, 13 % at worst (700x4096x512 10.3 / 11.7).
//   * up to 128 tokens and more than 128 outputs: one byte, always (65x136x4096 12.0 / 9.1, 120x4096x4096 17.9 / 13.3);
//   * up to 128 outputs the other side is the one-CTA kernel, whose tiles have 64 or 128 columns: 0.5 us a k-block, but
//     2 us less start (65x8x128 4.4 / 5.9, 512x64x256 5.8 / 6.0, 900x64x512 6.7 / 6.6, 1280x8x1024 8.5 / 9.1, 2000x8x1024 9.5 / 10.2,
//     2000x128x1024 11.8 / 9.6);
//   * rows of 2048 codes and more: one byte, but where tokens by the thousand fill two to five rounds of the packed side's
//     tiles to 0.82 or more, since the quantiser writes twice the bytes; with 256 columns a tile that counts below 4096 codes
//     only (tiles of 224: 2048x8192x8192 93.5 / 96.6, 1280x6144x4096 33.6 / 35.4; of 256: 1500x6144x2048 23.3 / 24.2, but
//     2048x6144x4096 46.8 / 46.2, 2600x6144x8192 102 / 88.8; not filled: 901x10240x8192 70.3 / 57.5, 1100x4096x4096 32.9 / 23.5;
//     more rounds: 8192x10240x8192 505 / 471);
//   * shorter rows: the estimate above against the packed side's, a round 0.43 us a k-block and 2.06, or 0.146 and 4.2 where
//     its epilogue sets the pace, and 5.5 us of start and end (6.05 up to 900 tokens, 7.0 there beyond 256 codes: with few
//     tiles its last one is rarely full).  Up to 900 tokens from 640 codes on one byte is ahead all through (2300x8192x128
//     22.5 / 25.9, 700x10240x256 14.5 / 15.8, 8192x14336x1024 136 / 145; 1100x1536x1024 12.5 / 10.3, 600x4096x256 9.4 / 8.5).
// All that is of the lightest epilogue.  `extras`: 1 with an asymmetric grid, factors of tokens or a residual, 2 with a residual
// on an asymmetric grid.  They cost this kernel more, whose threads hold four features of two tokens each: where the packed
// side's tiles are well filled, rows of up to 2048 codes (2: 3072; up to 900 tokens 512 and 1536) stay there (us: asymmetric
// 8192x28672x1280 270 / 331, dynamic 2048x14336x2048 52.4 / 58.1, residual 8192x10240x256 125 / 149, both 8192x4096x2048 76.4 / 88.3;
// not filled: asymmetric 1641x2776x3200 28.6 / 21.7, both 1003x1024x2048 14.5 / 10.5), and so do short rows that the estimates
// speak clearly against (residual 5356x576x640 12.4 / 13.6).  5000 calls: 0.3 % behind the better side, 17 % at worst
// (160x28672x128 with both 14.7 / 17.2).
inline bool wt_ahead(int M, int N, int K, int pairs, int extras) {
  if (M <= 64) return false;
  if (N <= 128) return K + 8 * N > (M <= 900 ? 768 : M <= 1500 ? 1152 : 1536);
  if (M <= 128) return true;
  const int tn = pair_tile_width(M, N, pairs);
  const long long tiles = (long long)((M + kPairRows - 1) / kPairRows) * ((N + tn - 1) / tn), rounds = (tiles + pairs - 1) / pairs;
  auto filled = [&](int percent) { return 100ll * M * N >= percent * rounds * pairs * kPairRows * tn; };
  const long long kblocks = K / 128, round = kblocks > 7 ? 430 * kblocks + 2060 : 146 * kblocks + 4200;
  auto ahead = [&](int start, int percent) {             // of the packed side's estimate, to that much of it
    return wt_cut(M, N, K, pairs, pairs * 4 / 9).ns * 100 <= (rounds * round + start) * percent;
  };
  if (extras > 0 && M > 900 && K <= (extras > 1 ? 3072 : 2048))
    return !filled(extras > 1 || K <= 512 ? 70 : 75) && (K >= 2048 || ahead(5500, 107));
  if (extras > 0 && M <= 900 && K <= (extras > 1 ? 1536 : 512) && filled(extras > 1 ? 60 : 65)) return false;
  if (K >= 2048) return M <= 900 || rounds < 2 || rounds > 5 || (K >= 4096 && tn == kPairWidth) || !filled(82);
  if (M <= 900 && K > 512) return true;
  return ahead(M > 900 ? 5500 : K <= 256 ? 6050 : 7000, 100);
}
// The same for the gate||up matmul of a SwiGLU block of more than 128 tokens (N = 2 d_ff).  The packed side's epilogue is
// slow with a ragged last tile, so that only many rounds of short rows are better there (blocks of tokens x d x d_ff, us:
// 8192x1024x4096 183 / 203, 4096x1024x4096 99.7 / 108; but 2048x1024x4096 68.0 / 65.6, 1500x2048x5632 90.9 / 74.9, 3000x4096x14336
// 390 / 359; 4096x2048x8192 215 / 221).
inline bool wt_ahead_swiglu(int M, int N, int K, int pairs) {
  const long long tiles = (long long)((M + kPairRows - 1) / kPairRows) * ((N + kPairWidth - 1) / kPairWidth);
  return M <= 900 || K >= 2048 || tiles <= 6ll * pairs;
}

}  // namespace fpt
