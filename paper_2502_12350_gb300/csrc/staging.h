// Page-locked staging of a context's uploads, so that the host neither waits for
// each copy nor keeps the vectors.  No CUDA types (tests/test_device_state.py).
#pragma once

#include <algorithm>
#include <cstddef>

namespace mamute {

// What a call stages is counted, and begin(), which starts a call, makes room for
// as much, up to kMax; what does not fit is copied from the vector and waited for.
// kMax: larger tables take long to plan, beside which the waits do not show
// (gradient calls with 17, 62 and 125 MB of tables take 14.2, 57 and 118 ms with
// 16 MB staged, and 14.4, 57 and 124 with all of it).
class Staging {
 public:
  static constexpr size_t kMax = 16u << 20;

  // Starts a call: wait() for copies of a failed call that may still be in flight
  // (zero on success), then alloc(bytes) (null: none to be had) and free(p).
  template <typename Wait, typename Alloc, typename Free>
  int begin(Wait wait, Alloc alloc, Free free) {
    const int e = used_ > 0 ? wait() : 0;
    const size_t want = std::min(need_, kMax);
    if (want > bytes_) {
      release(free);
      p_ = static_cast<char*>(alloc(want));
      bytes_ = p_ ? want : 0;
    }
    used_ = need_ = 0;
    return e;
  }

  // Room for `bytes`, or null.
  void* take(size_t bytes) {
    const size_t room = (bytes + 255) / 256 * 256;
    need_ += room;
    if (used_ + room > bytes_) return nullptr;
    void* p = p_ + used_;
    used_ += room;
    return p;
  }

  template <typename Free>
  void release(Free free) {
    if (p_) free(p_);
    p_ = nullptr;
    bytes_ = 0;
  }

  size_t bytes() const { return bytes_; }

 private:
  char* p_ = nullptr;
  size_t bytes_ = 0, used_ = 0, need_ = 0;
};

}  // namespace mamute
