// What the host remembers about a CUDA device.  No CUDA types, so that the
// rules are tested on the host (tests/test_device_state.py).
#pragma once

#include <algorithm>
#include <array>
#include <atomic>
#include <cstddef>
#include <map>
#include <mutex>

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

// The dynamic shared memory that one kernel has been allowed, per device: the
// allowance is an attribute of the kernel on a device, and setting it again may
// lower it under a launch of another thread.  raise() sets it through
// set(bytes), zero on success, where it is not yet that large.
class SmemLimit {
 public:
  template <typename F>
  int raise(int device, size_t bytes, F set) {
    const bool shared = device < 0 || device >= kDevices - 1;  // the last entry is of all others
    std::atomic<size_t>& have = have_[shared ? kDevices - 1 : device];
    if (!shared && have.load(std::memory_order_acquire) >= bytes) return 0;
    std::lock_guard<std::mutex> lock(mutex_);
    const size_t old = have.load(std::memory_order_relaxed);
    if (!shared && old >= bytes) return 0;
    const size_t want = std::max(old, bytes);
    const int e = set(want);
    if (e == 0) have.store(want, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::mutex mutex_;
  std::atomic<size_t> have_[kDevices] = {};
};

}  // namespace mamute
