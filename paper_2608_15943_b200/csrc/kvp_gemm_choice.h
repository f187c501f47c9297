// Which of the library's kernels a forward GEMM (K-major operands, one segment) runs on, and with which tiles (no CUDA
// dependency: a host-only test uses the same rules).
#pragma once

#include <math.h>

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
  int stages;
};

// Up to SPLIT_MAX_ROWS rows: tokens per tile and K split by an estimate of the time (us), whose constants were fitted to 1100
// launches (15 weight shapes x 9 row counts, weights not in L2, each behind an element-wise kernel, replayed from a graph;
// the choice it makes costs 0.5 % more than the best of all on average).  A CTA's k-blocks and the memory both count, as the
// root of the sum of their squares; a cluster costs up to a microsecond, and clusters of eight do not all fit at once from
// about seven tenths of the SMs on; more CTAs than SMs share them in twos, with half the ring.  The smallest split that gave
// 128 CTAs, with all tokens in one tile, was 15 % slower on average (16 x 2048 x 2048 13.4 us -> 8.2, 16 x 2048 x 5504 15.4 ->
// 9.7, 128 x 1024 x 1024 9.4 -> 6.7, 128 x 5504 x 2048 15.0 -> 11.4).
inline SplitConfig split_config(const GemmSize* probs, int n, int sms) {
  int rows = 0, columns = 0, deepest = 0, shallowest = 1 << 30;
  float weights = 0.f;
  for (int i = 0; i < n; ++i) {
    const int kb = (probs[i].K + GEMM_BK - 1) / GEMM_BK;
    rows = std::max(rows, probs[i].M);
    columns += (probs[i].N + SPLIT_COLS - 1) / SPLIT_COLS;
    deepest = std::max(deepest, kb);
    shallowest = std::min(shallowest, kb);
    weights += 2.f * probs[i].N * probs[i].K;
  }
  auto up = [](int x, int y) { return (x + y - 1) / y; };
  SplitConfig best{0, 1, 0};
  float best_us = 1e30f;
  int ctas = 0;
  for (int tok_tiles = 1; tok_tiles <= 4; tok_tiles *= 2) {
    const int nt = up(up(rows, tok_tiles), 16) * 16, tiles = columns * tok_tiles;
    if (up(rows, nt) != tok_tiles) continue;
    for (int split = 1; split <= 8; split *= 2) {
      if (split > 1 && 2 * split > shallowest) break;
      if (tiles * split > (tok_tiles == 1 && split < 8 ? 2 * sms : sms) && (tok_tiles > 1 || split > 1)) break;
      const float over = std::max(0.f, float(tiles * split) / sms - 1.f);   // CTAs that share an SM
      const float main = up(deepest, split) * (0.144f + 0.017f * nt / 128.f) * (1.f + 3.7f * over), memory = weights / 7.2e6f;
      const float cluster = split == 1 ? 0.f : split == 2 ? 0.6f : split == 4 ? 0.83f : 10 * tiles * split > 7 * sms ? 6.6f : 0.88f;
      const float us = sqrtf(main * main + memory * memory) + 0.0277f * nt + cluster + 0.098f * nt * over;
      if (us >= best_us) continue;
      best_us = us;
      best.nt = nt;
      best.split = split;
      ctas = tiles * split;
    }
  }
  const int ring_bytes = (ctas <= sms ? 220 : 110) * 1024;
  best.stages = std::min(SPLIT_MAX_STAGES, ring_bytes / (SPLIT_B_BYTES + best.nt * GEMM_BK * 2));
  return best;
}

// ------------------------------------------------------------------------------------------------------------
// Which kernel a forward GEMM of more than 128 rows runs on.  The times (us) of each are estimated from a model with the
// terms that bound it -- launches and tiles at fixed cost, an SM's share of L2 bandwidth, the tensor pipe, memory -- whose
// constants were fitted to 3400 measurements (11 weight shapes x 28 row counts, weights not in L2).  The choice it makes
// costs 0.7 % more than the best of all choices on average, CTA pairs always 50 %.  From PAIR_ROUNDS rounds of pair tiles on
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
    if (nt > 224) continue;   // (longer tiles draw more from L2 than the model says: 900 x 4096 x 11008 76 us for 65)
    consider(Choice::kSplit, nt, split, 4.7f + std::max(float(kb) / split * 0.11f * (1.f + nt / 128.f), (weights + rows) / 9.6e6f) +
                                                   0.027f * nt + (split > 1 ? 0.75f : 0.f));
  }
  return best;
}

}  // namespace kvp
