// How the attention backward is cut into CTAs, and their order (no CUDA dependency: a host-only test uses the same rules).
// A step is one 64-row query tile of one query stream (layer, query head) against one 128-row key tile.
#pragma once

#include <math.h>

#include <algorithm>

namespace kvp {

constexpr int BWD_KEYS = 128;      // key rows per tile
constexpr int BWD_QUERIES = 64;    // query rows per step
// A CTA's window of query tiles is sized so that it runs about this many steps (window x streams): long enough
// to amortise its prologue and its dK / dV reduction, short enough that a wave's footprint stays in L2.
constexpr int kStepsPerCta = 256;
constexpr int kMinWindow = 16;
// A CTA costs about seven steps besides its steps (prologue, dK / dV reduction, gap between two CTAs), and the last CTAs of
// a launch leave the device idle for some part of their length: with n steps per SM in all, n * 7 / t + 0.3 t is least at
// t = sqrt(24 n), and there is nothing to gain from fewer CTAs than one for every SM (1.5 n).  Fitted, like the order below, when a
// step took 1830 cycles at either head size; at heads of 64, where it now takes about a quarter less, a CTA's cost is more steps.
// Measured (bwd_kernel, us; always 256 steps -> this, in the order below): B3 S776 H16/4 dh64, 3 layers 120 -> 79; B4 S632
// H8/2 dh128, 8 layers 128 -> 107; B1 S2048 H8/8 dh128, 1 layer 51 -> 42; B1 S4096 H32/8 dh128, 1 layer 458 -> 351.  From
// about 2700 steps per SM on the 256 stand.
constexpr float kTailFactor = 24.f;
constexpr int kMinSteps = 2;

struct BwdCut {
  int window = 1;   // query tiles per CTA
  int parts = 1;    // parts the query streams of a (window, key tile) are dealt out in
};

struct BwdSizes {
  int n_jt, n_qt;          // key tiles, query tiles
  int n_pairs;             // (batch, KV head)
  int G;                   // query heads per KV head
  bool causal;
  int sms;
};

// Windows first (a CTA that serves all streams of its window loads K and V once for them), then parts of the streams where
// even the smallest window holds more steps than a CTA should run.
inline BwdCut bwd_cut(const BwdSizes& z, int streams, int target) {
  BwdCut c;
  int window = std::max(std::max(1, target / (kStepsPerCta / kMinWindow)), (target + streams - 1) / streams);
  if (window > 1) window += window & 1;   // whole key tiles of two query tiles: no CTA for half of a diagonal tile
  c.window = std::min(z.n_qt, window);
  c.parts = target < kStepsPerCta ? std::max(1, std::min(streams, (streams * c.window + (c.window == 1 ? target - 1 : target / 2)) / target)) : 1;
  // Up to 128 tokens dQ has one term, and two CTAs' terms of dK / dV add up to the same value in either order: such short
  // sequences keep results that do not differ from run to run.
  if (z.n_jt == 1) c.parts = std::min(c.parts, c.window < z.n_qt ? 1 : 2);
  return c;
}

inline double bwd_steps_per_sm(const BwdSizes& z, int layers) {
  long long stream_steps = 0;      // of one query stream of one (batch, KV head)
  for (int j = 0; j < z.n_jt; ++j) stream_steps += z.causal ? z.n_qt - j * (BWD_KEYS / BWD_QUERIES) : z.n_qt;
  return double(stream_steps) * z.n_pairs * layers * z.G / z.sms;
}

// The steps one CTA should run, with n steps per SM in all.
inline int bwd_target_steps(double n) {
  return std::max(kMinSteps, int(std::min(std::min(float(kStepsPerCta), 1.5f * float(n)), sqrtf(kTailFactor * float(n)))));
}

// CTAs longest first, so that the short ones (diagonal key tiles, last windows, small groups) fill in at the end, or in index
// order, which keeps what a wave touches in L2?  The former as long as Q, dO and the dQ accumulators of the launch about fit
// L2 in any order, and for so many steps per SM; a mask makes the CTAs differ more.  Measured over 920 shapes (longest first
// / index order, geometric mean, worst): causal up to 200 MB and 256 steps 0.95, 256 to 512 steps 1.02; 200 to 300 MB 1.02,
// 1.28; above 1.09, 1.30 (8 x 1024 tokens, 32 heads on 8 of 128, four layers: 1.1 GB, 498 steps, 1110 -> 1410 us); without
// a mask up to 200 MB and 128 steps 0.995, 128 to 256 steps 1.03, above 200 MB 1.06, 1.30.
constexpr double kFitsL2 = 200e6, kLongestFirst = 256., kLongestFirstFull = 128.;
inline bool bwd_longest_first(const BwdSizes& z, int layers, double steps_per_sm, long long q_rows, int dh) {
  return steps_per_sm <= (z.causal ? kLongestFirst : kLongestFirstFull) && 8. * double(q_rows) * dh * layers <= kFitsL2;
}

}  // namespace kvp
