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

// A launch's time in units of a key tile of a work item (two query tiles): the average over the SMs, but no less than the
// longest item.  An item costs one unit besides its key tiles, and an item of one query tile 0.6 of a unit for each.
struct FwdTime {
  float average, longest;
  float total() const { return std::max(average, longest); }
};
inline FwdTime fwd_time(const FwdSizes& z, int pack) {
  const int rows = FWD_ROWS >> pack, tiles = (z.S + rows - 1) / rows;
  auto key_tiles = [&](int t) { return ((z.causal ? std::min(z.S, (t + 1) * rows) : z.S) + FWD_ROWS - 1) / FWD_ROWS; };
  float sum = 0.f, longest = 0.f;
  for (int t = 0; t + 1 < tiles; t += 2) {
    const float cost = 1.f + 0.5f * (key_tiles(t) + key_tiles(t + 1));
    sum += cost;
    longest = std::max(longest, cost);
  }
  if (tiles & 1) {
    const bool by_heads = fwd_odd_by_heads(z, pack);
    const float cost = 1.f + (by_heads ? 1.f : 0.6f) * key_tiles(tiles - 1);
    sum += by_heads ? 0.5f * cost : cost;
    longest = std::max(longest, cost);
  }
  return FwdTime{sum * float(z.kv_heads * (z.G >> pack)) / z.sms, longest};
}

// Tiles of several heads waste less on the last, part-filled tile of a sequence and on the keys that a causal mask hides from
// a tile's first rows; both matter for short sequences only, and where the launch has fewer items than SMs an item's own time
// counts.  With a mask the two tiles of an item also walk the same number of key tiles, which gains at heads of 64 where the
// estimate says that nothing changes, if there are items enough.  At heads of 128 and without a mask the packed kernel itself
// takes up to a tenth longer for the same key tiles (long launches, against the estimate: causal heads of 64 1.00, full
// attention 1.05 to 1.08, heads of 128 1.02 to 1.05 up to 1200 tokens and 1.09 beyond), so that there it has to save an eighth.
// Measured on 1660 shapes of 8 to 3000 tokens (heads packed / not, geometric mean of those where this says so): launches of up to
// a millisecond 0.79, 2 % of them more than 3 % slower, 1.08 at most; longer ones 0.95, 1.04 at most; 3 x 776 tokens, 16 heads of
// 64 on 4, three layers 35.2 -> 31.3 us.  One line at 0.97 for all of them slowed long launches at heads of 128 by 6 % on
// average and 19 % at most (9 x 2032 tokens, 64 heads on 8, four layers, 2.33 -> 2.78 ms).
constexpr int FWD_PACK_TOKENS = 2048;
inline int fwd_pack(const FwdSizes& z) {
  const int pack = fwd_most_pack(z.G);
  if (pack == 0 || z.S > FWD_PACK_TOKENS) return 0;
  const FwdTime heads = fwd_time(z, pack), head = fwd_time(z, 0);
  if (!z.causal || z.dh > 64) return heads.total() < 0.88f * head.total() ? pack : 0;
  const bool even = heads.average > (z.S < 1024 ? 1.4f : 1.f) * heads.longest && heads.total() <= head.total();
  return heads.total() < 0.97f * head.total() || even ? pack : 0;
}

}  // namespace kvp
