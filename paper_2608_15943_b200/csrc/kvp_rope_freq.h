// Frequencies of the rotary embedding (no CUDA dependency: a host-only test uses the same function).
#pragma once

#include <math.h>

namespace kvp {

// theta^(-2i/dh), i < dh / 2, as float pairs hi + lo, which hold a value to 2^-48.  By repeated multiplication, one power
// instead of one for every pair (3 us of a 13 us call): in long double (64 bits of mantissa), where i roundings and the
// i-fold error of the ratio stay below 2^-55 for 128 pairs.  (In double they came to 2^-47.)
inline void rope_frequencies(double theta, int dh, float* hi, float* lo, int stride) {
  const long double ratio = powl((long double)theta, -2.0L / dh);
  long double f = 1.0L;
  for (int i = 0; i < dh / 2; ++i, f *= ratio) {
    hi[i * stride] = float(f);
    lo[i * stride] = float(f - (long double)hi[i * stride]);
  }
}

}  // namespace kvp
