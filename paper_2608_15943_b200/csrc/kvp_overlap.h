// Do the outputs of a call share memory with its inputs?  (No CUDA dependency: a host-only test uses the same code.)
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>
#include <initializer_list>
#include <utility>
#include <vector>

namespace kvp {

struct Tensors {            // one per-layer array of an entry point
  const void* const* at;
  size_t bytes;             // of each tensor
  const int32_t* donor;     // not null: only the owners' entries are tensors
  bool is(int l) const { return donor == nullptr || donor[l] == l; }
  uintptr_t from(int l) const { return reinterpret_cast<uintptr_t>(at[l]); }
};

// Where a call writes: tensors that do not share memory with one another.  As a rule no input lies between the first and the last of
// them, and that is all it takes; else they are sorted, and searched for the input.
class Outputs {
 public:
  Outputs(int L, std::initializer_list<Tensors> outs) : L_(L) {
    at_.reserve(outs.size() * size_t(L));
    for (const Tensors& t : outs)
      for (int l = 0; l < L; ++l)
        if (t.is(l)) {
          const Range r{t.from(l), t.from(l) + t.bytes};
          all_ = Range{std::min(all_.first, r.first), std::max(all_.second, r.second)};
          at_.push_back(r);
        }
  }
  // Any of them with any tensor of `in`; `own`: apart from those in the place of that layer's tensor of `own`, an output.
  bool meet(const Tensors& in, const Tensors* own = nullptr) {
    for (int l = 0; l < L_; ++l) {
      if (!in.is(l) || in.from(l) >= all_.second || in.from(l) + in.bytes <= all_.first || (own != nullptr && own->at[l] == in.at[l])) continue;
      if (!sorted_) std::sort(at_.begin(), at_.end());
      sorted_ = true;
      auto next = std::lower_bound(at_.begin(), at_.end(), in.from(l), [](const Range& o, uintptr_t x) { return o.second <= x; });
      if (next != at_.end() && next->first < in.from(l) + in.bytes) return true;
    }
    return false;
  }

 private:
  using Range = std::pair<uintptr_t, uintptr_t>;
  int L_;
  bool sorted_ = false;
  Range all_{UINTPTR_MAX, 0};
  std::vector<Range> at_;
};

}  // namespace kvp
