// sdv_sets.h - which of a workspace's two sets of tile partials a call uses (host only).
#pragma once

#include <cstddef>
#include <cstdint>
#include <mutex>

namespace sdv {

// Calls on a workspace use its two sets in turn, remembered for the last kSlots workspaces.
// Where set 1 starts depends on the call's sizes, so that a call of another layout may have
// written anywhere in both sets: a change of layout, like a workspace that is not remembered,
// makes both of them fresh.  The first call on a fresh set waits for the previous kernel
// before it stores a partial.
class PartialSets {
 public:
  static constexpr size_t kSlots = 64;

  // The set (0 or 1) of the next call on `workspace`; *fresh: it is not known to hold the
  // partials of this layout only.
  int next(const void* workspace, uint64_t layout, bool* fresh) {
    std::lock_guard<std::mutex> lock(mu_);
    Entry& e = tab_[(reinterpret_cast<uintptr_t>(workspace) >> 8) % kSlots];
    if (e.ws != workspace || e.layout != layout) e = Entry{workspace, layout, 0, {false, false}};
    const int set = e.next;
    *fresh = !e.used[set];
    e.used[set] = true;
    e.next ^= 1;
    return set;
  }

 private:
  struct Entry {
    const void* ws;
    uint64_t layout;
    int next;
    bool used[2];
  };
  std::mutex mu_;
  Entry tab_[kSlots] = {};
};

}  // namespace sdv
