// Do per-layer arrays of a call share memory?  (No CUDA dependency: a host-only test uses the same code.)
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace kvp {

struct Tensors {            // one per-layer array of an entry point
  const void* const* at;
  size_t bytes;             // of each tensor
  const int32_t* donor;     // not null: only the owners' entries are tensors
};

// Any tensor of `a` with any of `b`, of L layers; apart from a layer's two that are one (same_layer).  The arrays' bounds decide as a rule: each is one allocation, or they lie one
// after the other.
inline bool share_memory(int L, const Tensors& a, const Tensors& b, bool same_layer = false) {
  auto is = [](const Tensors& t, int l) { return t.donor == nullptr || t.donor[l] == l; };
  auto from = [](const Tensors& t, int l) { return reinterpret_cast<uintptr_t>(t.at[l]); };
  struct Bounds {
    uintptr_t lo, hi;
  };
  auto bounds = [&](const Tensors& t) {
    Bounds x{UINTPTR_MAX, 0};
    for (int l = 0; l < L; ++l)
      if (is(t, l)) x = Bounds{std::min(x.lo, from(t, l)), std::max(x.hi, from(t, l) + t.bytes)};
    return x;
  };
  const Bounds x = bounds(a), y = bounds(b);
  if (x.lo >= y.hi || y.lo >= x.hi) return false;
  for (int i = 0; i < L; ++i)
    for (int j = 0; j < L; ++j)
      if (is(a, i) && is(b, j) && !(same_layer && i == j && a.at[i] == b.at[j]) && from(a, i) < from(b, j) + b.bytes && from(b, j) < from(a, i) + a.bytes) return true;
  return false;
}

}  // namespace kvp
