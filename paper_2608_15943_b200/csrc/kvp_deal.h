// How a decode step's K/V rows are dealt out to blocks, in granules of 16 tokens (no CUDA dependency: the kernels, the host
// and a host-only test use the same rules).  `total`: granules of all units of the launch; a unit is one (donor group,
// sequence, KV head); `fit`: blocks that fit on the device.
#pragma once

#ifdef __CUDACC__
#define KVP_HD __host__ __device__
#else
#define KVP_HD
#endif

namespace kvp {

// (nearly all dividends fit 32 bits, and all divisors, where a division takes a fifth of the time)
KVP_HD inline long long div_places(long long a, long long b) {
  return (a | b) >> 32 == 0 ? (long long)(unsigned(a) / unsigned(b)) : a / b;
}

constexpr int MIN_SHARE = 8;       // places of a share at least: a piece costs a block about as much again
// Places of a share at least where there are more shares than blocks that fit, and shares per block that fits at most.  (At
// dh 64 four blocks share an SM, so that starting one costs little: 64 sequences of 100 to 6400 tokens, 8 KV heads, three
// groups 225 us with 160 and 16, 217 so.  The grid holds the shares of the longest list the block table allows, and blocks
// beyond the actual ones cost time too: 16 sequences of 4096 tokens in a table for 131072 32 us with 5, 36 with 8.)
KVP_HD constexpr int long_share(int dh) { return dh == 64 ? 80 : 160; }
KVP_HD constexpr int max_rounds(int dh) { return dh == 64 ? 5 : 16; }

// Whole units are dealt out where they are short on average, since every piece costs a block a merge of its warps: up to 32
// granules; up to 512 KB where there are units enough for three quarters of the blocks; at dh 64 (granules of 4 KB) up to 64
// for a quarter of them.  But the longest must not keep its block busy for much longer than an equal share would: one long
// sequence among short ones is cut.
KVP_HD inline bool dealt_by_units(int dh, long long total, long long units, long long longest, int fit) {
  const int many = 8192 / dh;
  const int most = 4 * units >= 3LL * fit ? many : dh == 64 && 4 * units >= fit ? 64 : 32;
  return total < most * units && (longest <= many || longest * fit <= 2 * total);
}

// Otherwise the units lie one behind the other, each with some empty places behind its granules that stand for its merge:
// a share of many short units then takes as long as one of a few long ones.  (None where every block gets as little as it
// may: there a share's latency counts.)  Measured (us, the mean length alone deciding and no empty places -> so; dh 128, 8 KV
// heads): 32768 tokens and 63 sequences of 300 310 -> 77, 30000 and 39 of 200 286 -> 61, 4 of 4096 and 28 of 64 in two groups
// 69 -> 47, 8000 and 3 of 50 30 -> 24.
KVP_HD inline int unit_rest(int dh, long long total, int fit) { return total / MIN_SHARE <= fit ? 0 : dh == 64 ? 16 : 12; }

// Shares a list of `places` is dealt out in.
KVP_HD inline int shares_for(int dh, int fit, int max_shares, long long places) {
  long long n = places / MIN_SHARE;
  if (n > fit) {
    const long long rounds = div_places(places, (long long)fit * long_share(dh));
    n = (long long)fit * (rounds < 1 ? 1 : rounds > max_rounds(dh) ? max_rounds(dh) : rounds);
  }
  return int(n < 1 ? 1 : n > max_shares ? max_shares : n);
}

}  // namespace kvp
