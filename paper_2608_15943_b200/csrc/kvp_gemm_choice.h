// Which of the library's kernels a forward GEMM (K-major operands, one segment) runs on, and with which tiles (no CUDA
// dependency: a host-only test uses the same rules).
#pragma once

#include <stdint.h>

#include <algorithm>

namespace kvp {

struct GemmSize {
  int M, N, K;
};

constexpr int GEMM_BK = 64;                      // depth of a k-block
constexpr int GEMM_BM = 128, GEMM_PAIR_BM = 256; // rows of a tile of the single-CTA and the CTA-pair kernel
constexpr int SPLIT_COLS = 128;                  // columns of a tile of the split kernel: the M of its MMA
constexpr int SPLIT_MAX_STAGES = 8;
// Tokens of a tile of the column-owning pairs: the N of an MMA with M = 256 on a CTA pair goes in steps of 32.
constexpr int TALL_UNIT = 32;
constexpr int SPLIT_B_BYTES = SPLIT_COLS * GEMM_BK * 2;
constexpr int SPLIT_MAX_ROWS = 128;       // up to here always the split kernel

struct SplitConfig {
  int nt;       // tokens per tile
  int split;    // CTAs of a cluster along K
  int parts;    // accumulators of a CTA, each with half of its k-blocks where there are two
  int stages;
};

// Up to SPLIT_MAX_ROWS rows.  K is cut into the smallest number of pieces that gives 128 CTAs, eight at most, each with an
// accumulator of its own: by the columns and the depth alone, so that a row's bits do not depend on how many rows the call has.
// Fewer pieces would be faster for many shapes, but the error of a tensor-core sum grows with its length: fp32 results of a
// split chosen by time alone, often a half or a quarter of this one, lay 2.4 times as far from 64 bits on average, 7.7 times
// at most, over the 442 of 720 shapes where it differed.
// A cluster takes the pieces, a CTA each.  Where the launch would put a CTA on nearly every SM, not all clusters find room at
// once (of eight CTAs from 13/16 of the SMs on, of four from 132 of 148): half as many CTAs with two accumulators take the
// pieces then.  The tokens go into two or four tiles where all CTAs still fit.  Measured (us, one tile and one CTA a piece ->
// this; weights not in L2, each launch behind an element-wise kernel, replayed from a graph): two accumulators, 16 x 2048 x
// 2048 10.6 -> 7.8, 128 x 2048 x 2048 16.0 -> 11.2, 64 x 4608 x 4096 18.9 -> 15.4; more tiles, 128 x 256 x 256 7.3 -> 5.2, 128 x
// 512 x 1024 7.9 -> 6.7.  On average over 15 weight shapes x 7 row counts 1.07 times as fast, over 31 other shapes 1.11, and 0.4 %
// above the best cluster, tile and number of accumulators for these pieces on both.
inline SplitConfig split_config(const GemmSize* probs, int n, int sms) {
  int rows = 0, columns = 0, kblocks = 1 << 30;
  for (int i = 0; i < n; ++i) {
    rows = std::max(rows, probs[i].M);
    columns += (probs[i].N + SPLIT_COLS - 1) / SPLIT_COLS;
    kblocks = std::min(kblocks, (probs[i].K + GEMM_BK - 1) / GEMM_BK);
  }
  auto tile = [&](int tiles) { return ((rows + tiles - 1) / tiles + 15) / 16 * 16; };
  SplitConfig c{tile(1), 1, 1, 0};
  while (c.split < 8 && 2 * c.split <= kblocks && columns * c.split < 128) c.split *= 2;
  int ctas = columns * c.split;
  auto fit = [&] { return c.split == 8 ? 13 * sms / 16 : c.split == 4 ? sms - 16 : sms; };
  if (ctas > fit() && ctas <= sms) {
    c.split /= 2;
    c.parts = 2;
    ctas /= 2;
  }
  for (int tiles = 2; tiles <= 4 && columns * c.split * tiles <= fit(); tiles *= 2) {
    if ((rows + tile(tiles) - 1) / tile(tiles) != tiles) break;
    c.nt = tile(tiles);
    ctas = columns * c.split * tiles;
  }
  const int ring_bytes = (ctas <= sms ? 220 : 110) * 1024;
  c.stages = std::min(SPLIT_MAX_STAGES, ring_bytes / (SPLIT_B_BYTES + c.nt * GEMM_BK * 2));
  return c;
}

// ------------------------------------------------------------------------------------------------------------
// Which kernel a forward GEMM of more than 128 rows runs on.  The times (us) of each are estimated from a model with the
// terms that bound it -- launches and tiles at fixed cost, an SM's share of L2 bandwidth, the tensor pipe, memory -- whose
// constants were fitted to 3400 measurements (11 weight shapes x 28 row counts, weights not in L2) before the split kernel's
// sum and the tile kernels' stores were shortened.  On the kernels as they are the choice costs 0.6 % more than the best of all
// choices on average over 15 weight shapes x 14 row counts (11 % at most; CTA pairs always 38 %), 1.2 % over 31 shapes that
// the fit never saw (10 %; 52 %).  From PAIR_ROUNDS rounds of pair tiles on
// and above 4096 rows the pairs' order of tiles (an A slab stays in L2) counts, and they stand: 3000 rows x 32000 x 4096 508
// us on them, 597 in tiles of one size.
// ------------------------------------------------------------------------------------------------------------
constexpr int PAIR_ROUNDS = 16;
constexpr int CHOICE_MAX_ROWS = 4096;
struct Choice {
  enum Kind { kSingle, kPair, kTall, kSplit } kind = kPair;
  int nt = 0;         // tokens per tile (tall, split)
  int split = 1;
  float us = 1e30f;
};

inline Choice choose_forward(const GemmSize* probs, int n, int sms) {
  int M = 0, kb = 0, shallowest = 1 << 30, cols128 = 0, cols256 = 0;
  float weights = 0.f, rows = 0.f;   // bytes of B, of A and C
  for (int i = 0; i < n; ++i) {
    const GemmSize& g = probs[i];
    M = std::max(M, g.M);
    kb = std::max(kb, (g.K + GEMM_BK - 1) / GEMM_BK);
    shallowest = std::min(shallowest, (g.K + GEMM_BK - 1) / GEMM_BK);
    cols128 += (g.N + 127) / 128;
    cols256 += (g.N + 255) / 256;
    weights += 2.f * g.N * g.K;
    rows += 2.f * g.M * g.N + (i == 0 ? 2.f * g.M * g.K : 0.f);
  }
  const int pairs = sms / 2;
  Choice best;
  if ((M + GEMM_PAIR_BM - 1) / GEMM_PAIR_BM * cols256 > PAIR_ROUNDS * pairs) return best;
  auto consider = [&](Choice::Kind kind, int nt, int split, float us) {
    if (us >= best.us) return;
    best.kind = kind;
    best.nt = nt;
    best.split = split;
    best.us = us;
  };
  auto up = [](int x, int y) { return (x + y - 1) / y; };
  const float memory = (weights + rows) / 5.95e6f;
  consider(Choice::kSingle, 0, 1, 2.3f + std::max(up(up(M, GEMM_BM) * cols256, sms) * (kb * 0.361f + 4.3f), memory));
  consider(Choice::kPair, 0, 1, 3.2f + std::max(up(up(M, GEMM_PAIR_BM) * cols256, pairs) * (kb * 0.338f + 4.3f), memory));
  // column-owning pairs, tiles of equal size along the tokens
  const int fewest = up(M, 256);
  for (int k = fewest; k < fewest + 4 + fewest / 3; ++k) {
    const int nt = up(up(M, k), TALL_UNIT) * TALL_UNIT;
    if (k > fewest && nt < 80) break;
    const float tile = kb * std::max(0.157f * (1.f + nt / 256.f), 0.00139f * nt) + 2.5f;
    consider(Choice::kTall, nt, 1, 3.7f + std::max(up(up(M, nt) * cols256, pairs) * tile, memory));
  }
  // split kernel: one CTA per SM; clusters of four do not fill every GPC; every CTA has k-blocks of every problem
  for (int split = 1; split <= 4 && 2 * split <= shallowest; split *= 2) {
    const int most = (split == 4 ? sms - 16 : sms) / (split * cols128);   // token tiles that fit
    if (most < 1) break;
    const int nt = std::max(48, up(up(M, most), 16) * 16);
    if (nt > 224) continue;   // (longer tiles draw more from L2 than the model says: 1000 x 4096 x 11008 82 us for 74)
    consider(Choice::kSplit, nt, split, 4.7f + std::max(float(kb) / split * 0.11f * (1.f + nt / 128.f), (weights + rows) / 9.6e6f) +
                                                   0.027f * nt + (split > 1 ? 0.75f : 0.f));
  }
  return best;
}

// ------------------------------------------------------------------------------------------------------------
// Up to 128 rows: are the weights read with the policy evict_first?  From 32 MB on, with one tile of tokens.  Where more passes
// between two uses of the same weights than L2 keeps, lines that leave first leave some of the others in place.  Measured (us,
// without -> with): token steps of two layers of d 4096, 1, 8 and 64 sequences 182.6 -> 173.3, 190.3 -> 184.0, 253.2 -> 250.2, of four
// layers, 16 sequences 531.1 -> 529.3 (the latter of the size of the noise); a head of 64 MB behind a layer of d 1024 61.8 ->
// 58.0.  Prefill of layers of d 4096, three sets of weights in turn (one set): one layer, 96 tokens 22.0 -> 20.4 (18.4 -> 18.6), three,
// 104 tokens 37.4 -> 35.9 (38.0 -> 35.2), five with few heads 30.5 -> 27.5 (29.5 -> 26.0); six of 128 tokens 72.9 -> 75.7, but 102 -> 89
// on new weights, when L2 is full of what wrote them.
// A training step of as few tokens reads its weights again in the backward, out of L2 where they are few: one layer of 96 tokens
// 74.2 -> 76.2, two of 72 102.6 -> 107.4, but three of 104 149.8 -> 144.7, four of 64 166.7 -> 164.1; with output projections 0.98 to
// 1.02 of the time.  A launch cannot tell one from the other, and prefill gains more.  Where the same weights come again at once:
// 4096 x 11008 at 1 and 32 rows 11.3 -> 12.3 to 14.1, 12.1 -> 12.7 to 14.9, three of 4096 x 4096 in turn 7.7 -> 8.0 each; one or two of
// them nothing, and 11008 x 4096 and four or more of 4096 x 4096 gain (18.1 -> 16.1 at 32 rows, 34.4 -> 31.9).
// At 160 rows it gains nothing (eight of 11008 x 4096 168.4 -> 168.4), and loads with a policy of any kind slow tiles that share
// B (1155 x 1024 x 2816 11.1 -> 12.2).
// ------------------------------------------------------------------------------------------------------------
constexpr double SPLIT_STREAM_BYTES = 32 * 1024 * 1024;
inline bool stream_weights(const GemmSize* probs, int n, int nt) {
  double bytes = 0;
  for (int i = 0; i < n; ++i) {
    if (probs[i].M > std::min(nt, SPLIT_MAX_ROWS)) return false;
    bytes += 2. * probs[i].N * probs[i].K;
  }
  return bytes >= SPLIT_STREAM_BYTES;
}

// ------------------------------------------------------------------------------------------------------------
// The tiles of a launch of gradient GEMMs, dealt out to CTA pairs.  They come in classes of equal cost, the costliest first:
// input gradients run over all columns of the weights (96 k-blocks and more), weight gradients over the tokens (a few).  Each
// class goes to the pairs so that the fullest of them is as empty as can be, a run of consecutive tiles to each.  Only where the
// costliest are fewer than the pairs: elsewhere every pair has some, and tiles taken in turn share more in L2 (2048 tokens, d
// 4096 153 us in turn, 157 dealt out).  Measured (us, in turn -> dealt out): 264 tokens, 7 layers of d 1024, 4096 + 2 x 1024 columns
// 80.5 -> 74.7; 1200 tokens, d 2048, 2048 + 2 x 1024 columns 43.6 -> 39.7.
// ------------------------------------------------------------------------------------------------------------
constexpr int DEAL_CLASSES = 6, DEAL_PAIRS = 96;

// Estimated time (us) of a tile of nt rows: its k-blocks at a pair's share of L2, or its stores at a pair's share of memory.
inline float gradient_tile_us(int kblocks, int nt, bool f32) {
  return std::max(kblocks * 0.157f * (1.f + nt / 256.f), (f32 ? 3.f : 1.5f) * nt / 256.f) + 0.6f;
}

// first[c][p]: the first tile of class c (tiles counted through all classes) that pair p takes, up to first[c][p + 1].
inline void deal_tiles(const float* cost, const int* tiles, int n_classes, int pairs, uint16_t (*first)[DEAL_PAIRS + 1]) {
  float load[DEAL_PAIRS] = {};
  int at = 0;
  for (int c = 0; c < n_classes; ++c) {
    const float per = cost[c], inv = 1.f / per;
    auto fits = [&](float level, int p) { return int(std::max(0.f, level - load[p]) * inv); };
    auto all = [&](float level) {
      int n = 0;
      for (int p = 0; p < pairs; ++p) n += fits(level, p);
      return n;
    };
    float sum = 0.f, most = 0.f;
    for (int p = 0; p < pairs; ++p) {
      sum += load[p];
      most = std::max(most, load[p]);
    }
    // between `low`, where the pairs do not take all tiles, and `high`, where they do
    float low = 0.f, high = std::max(most, (sum + tiles[c] * per) / pairs) + 1.01f * per;
    for (int i = 0; i < 16; ++i) {
      const float level = 0.5f * (low + high);
      (all(level) < tiles[c] ? low : high) = level;
    }
    int rest = tiles[c];
    for (int p = 0; p < pairs; ++p) rest -= fits(low, p);
    for (int p = 0; p < pairs; ++p) {
      int n = fits(low, p);
      const int more = std::min(rest, fits(high, p) - n);
      n += more;
      rest -= more;
      first[c][p] = uint16_t(at);
      at += n;
      load[p] += n * per;
    }
    first[c][pairs] = uint16_t(at);
  }
}

}  // namespace kvp
