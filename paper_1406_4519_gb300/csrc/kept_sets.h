// kept_sets.h -- resources of destroyed handles kept for the next ones, by CUDA
// context.
//
// A stream belongs to the context it was made in.  A device can have several
// contexts at a time or, after a reset, one after another, so what is kept is
// found by the context's id, which no later context of the process gets again,
// and never by the device's number.  Free of CUDA (a host-only test compiles it).
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <mutex>
#include <utility>
#include <vector>

namespace dfacto {

template <class Set>
class KeptSets {
 public:
  static constexpr size_t kPerContext = 32;
  static constexpr size_t kInAll = 256;  // sets of contexts that are gone stay until the process ends

  // Hand out a kept set of context `ctx`.  False if there is none.
  bool take(uint64_t ctx, Set* out) noexcept {
    try {
      std::lock_guard<std::mutex> g(mu_);
      for (size_t i = sets_.size(); i-- > 0;) {
        if (sets_[i].first != ctx) continue;
        *out = sets_[i].second;
        sets_[i] = sets_.back();
        sets_.pop_back();
        return true;
      }
    } catch (...) {
    }
    return false;
  }

  // Keep an idle set of context `ctx`.  False if it is not kept (the caller
  // destroys it).
  bool give(uint64_t ctx, const Set& s) noexcept {
    try {
      std::lock_guard<std::mutex> g(mu_);
      size_t same = 0;
      for (const auto& e : sets_) same += e.first == ctx;
      if (same >= kPerContext || sets_.size() >= kInAll) return false;
      sets_.emplace_back(ctx, s);
      return true;
    } catch (...) {
      return false;
    }
  }

 private:
  std::mutex mu_;
  std::vector<std::pair<uint64_t, Set>> sets_;
};

}  // namespace dfacto
