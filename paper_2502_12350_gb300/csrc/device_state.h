// What the host remembers about a CUDA device.  No CUDA types, so that the
// rules are tested on the host (tests/test_device_state.py).
#pragma once

#include <array>
#include <map>

namespace mamute {

// Resident blocks per SM of the kernel variants of one thread (a driver query of
// about a microsecond, asked for every candidate of every plan).  The key holds
// the device; a query that fails (negative) is asked again the next time.
class OccupancyMemo {
 public:
  using Key = std::array<int, 7>;  // device, then the variant and its table length
  template <typename F>
  int get(const Key& key, F query) {
    const auto it = known_.find(key);
    if (it != known_.end()) return it->second;
    const int n = query();
    if (n < 0) return n;
    if (known_.size() >= 4096) known_.clear();
    known_.emplace(key, n);
    return n;
  }

 private:
  std::map<Key, int> known_;
};

}  // namespace mamute
