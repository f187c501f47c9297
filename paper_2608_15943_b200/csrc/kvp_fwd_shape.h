// Whose rows share a query tile of the attention forward (no CUDA dependency: a host-only test uses the same rules).
#pragma once

#include <algorithm>

namespace kvp {

constexpr int FWD_ROWS = 128;      // rows of a query tile, and keys of a key tile
constexpr int FWD_MAX_PACK = 4;    // log2 of the heads that share a tile at most

struct FwdSizes {
  int S, G;                // tokens; query heads per KV head
  int dh;
  bool causal;
  long long kv_heads;      // of the launch: layers x batch x KV heads
  int sms;
};

// The heads of a KV head read the same keys, so a tile may hold 128 >> pack tokens of each of 1 << pack heads.
inline int fwd_most_pack(int G) {
  int pack = 0;
  while (pack < FWD_MAX_PACK && G % (2 << pack) == 0) ++pack;
  return pack;
}
// The last of an odd number of whole-head tiles makes an item with the next head's, unless every tile has an SM to itself.
inline bool fwd_odd_by_heads(const FwdSizes& z, int pack) {
  const int tiles = (z.S + (FWD_ROWS >> pack) - 1) / (FWD_ROWS >> pack);
  return pack == 0 && z.G % 2 == 0 && z.kv_heads * z.G * ((tiles + 1) / 2) > z.sms;
}

// A launch's time in units of a key tile of a work item (two query tiles).  An item costs one unit besides its key tiles, and
// an item of one query tile 0.6 of a unit for each.  Up to FWD_ROUNDS rounds of items the list is dealt out as the kernel does it
// (longest first, rounds in alternating direction, one CTA per SM), and the fullest CTA counts; beyond, the average.
constexpr int FWD_ROUNDS = 6;
inline float fwd_time(const FwdSizes& z, int pack) {
  const int rows = FWD_ROWS >> pack, tiles = (z.S + rows - 1) / rows;
  const long long groups = z.kv_heads * (z.G >> pack);
  const bool by_heads = fwd_odd_by_heads(z, pack);
  // the list: the last of an odd number of tiles, then the pairs of tiles from the end of the sequence on
  const long long n_odd = tiles & 1 ? (by_heads ? groups / 2 : groups) : 0, n = n_odd + groups * (tiles / 2);
  auto key_tiles = [&](int t) { return ((z.causal ? std::min(z.S, (t + 1) * rows) : z.S) + FWD_ROWS - 1) / FWD_ROWS; };
  const float odd = n_odd > 0 ? 1.f + (by_heads ? 1.f : 0.6f) * key_tiles(tiles - 1) : 0.f;
  auto pair = [&](int k) { return 1.f + 0.5f * (key_tiles((tiles & ~1) - 2 - 2 * k) + key_tiles((tiles & ~1) - 1 - 2 * k)); };
  const int pairs = tiles / 2;
  const float longest = std::max(odd, pairs > 0 ? pair(0) : 0.f);
  if (n <= z.sms) return longest;
  const int sms = z.sms;
  if (n > (long long)FWD_ROUNDS * sms) {
    float sum = float(n_odd) * odd;
    for (int k = 0; k < pairs; ++k) sum += float(groups) * pair(k);
    return std::max(sum / float(sms), longest);
  }
  const int items = int(n), first = int(n_odd), per = int(groups);
  auto cost = [&](int i) { return i < first ? odd : pair((i - first) / per); };
  auto load = [&](int cta) {
    float sum = 0.f;
    for (int r = 0, at = 0; at < items; ++r, at += sms) {
      const int i = at + (r & 1 ? sms - 1 - cta : cta);
      if (i < items) sum += cost(i);
    }
    return sum;
  };
  // neighbouring CTAs differ only where the cost changes along the list, or the list ends
  float most = std::max(load(0), load(sms - 1));
  auto look = [&](int i) { most = std::max(most, load((i / sms) & 1 ? sms - 1 - i % sms : i % sms)); };
  for (int at = first; at <= items; at += per) {
    if (at > 0) look(at - 1);
    look(at);
  }
  return most;
}

// Tiles of several heads waste less on the last, part-filled tile of a sequence and on the keys that a causal mask hides
// from a tile's first rows; both matter for short sequences only.  At heads of 128 and without a mask the packed kernel
// itself takes up to a tenth longer for the same key tiles (long launches, against the estimate: causal heads of 64 1.00,
// full attention 1.05 to 1.08, heads of 128 1.02 to 1.05 up to 1200 tokens and 1.09 beyond), so that there it has to save an
// eighth.  Measured on 1660 shapes of 8 to 3000 tokens (heads packed / not, geometric mean of those where this says so):
// launches of up to a millisecond 0.76, 1.03 at most, longer ones 0.93, 0.99 at most, on 428 packed ones drawn afterwards
// 0.77, 1.03; 3 x 776 tokens, 16 heads of 64 on 4, three layers 35.2 -> 31.3 us.  One line at 0.97 for all of them slowed
// long launches at heads of 128 by 6 % on average and 19 % at most (9 x 2032 tokens, 64 heads on 8, four layers, 2.33 ->
// 2.78 ms); with the average over the SMs in the place of the fullest CTA, launches of one or two rounds lost up to 12 % (2
// x 203 tokens, 64 heads of 128 on 8, two layers).
constexpr int FWD_PACK_TOKENS = 2048;
inline int fwd_pack(const FwdSizes& z) {
  const int pack = fwd_most_pack(z.G);
  if (pack == 0 || z.S > FWD_PACK_TOKENS) return 0;
  return fwd_time(z, pack) < (z.causal && z.dh == 64 ? 0.97f : 0.88f) * fwd_time(z, 0) ? pack : 0;
}

}  // namespace kvp
