// thor_staging.h -- host memory through which a context's small uploads and results pass
// (grow-only; contents are not kept across a growth).  Page-locked where it can be had: one
// asynchronous copy instead of a staged one.  Where it cannot, ordinary memory does: a call is
// slower then, not refused.  Locking and unlocking takes some 0.3 ms, which a copy saves some 10 us
// of, so the first kPlain requests are served from ordinary memory (a context made for one tiny
// run: 0.14 ms, 0.48 with the lock) and the block grows by powers of two.
#pragma once

#include <cstddef>
#include <cstdlib>

namespace thor {

class HostStaging {
 public:
  using Lock = bool (*)(void**, std::size_t);  // page-locked allocation; false where there is none
  using Unlock = void (*)(void*);
  HostStaging(Lock lock, Unlock unlock, std::size_t max_locked) : lock_(lock), unlock_(unlock), max_(max_locked) {}
  HostStaging(const HostStaging&) = delete;
  HostStaging& operator=(const HostStaging&) = delete;
  ~HostStaging() {
    if (locked_) unlock_(locked_);
    std::free(plain_);
  }
  static constexpr int kPlain = 2;
  // Page-locked memory, or NULL beyond max_locked, for the first kPlain requests, or where it
  // cannot be had.  `drain` waits for the copies out of and into the block that a growth frees.
  template <class Drain>
  void* locked(std::size_t bytes, Drain drain) {
    if (bytes > max_) return nullptr;
    if (requests_ < kPlain) {
      ++requests_;
      return nullptr;
    }
    if (locked_cap_ >= bytes) return locked_;
    if (locked_) {
      drain();
      unlock_(locked_);
    }
    locked_ = nullptr;
    locked_cap_ = 0;
    std::size_t cap = 16384;
    while (cap < bytes) cap *= 2;
    if (cap > max_) cap = max_;
    if (!lock_(&locked_, cap)) return locked_ = nullptr;
    locked_cap_ = cap;
    return locked_;
  }
  // Page-locked memory, else ordinary memory; NULL only where there is no memory at all.
  template <class Drain>
  void* any(std::size_t bytes, Drain drain) {
    if (void* p = locked(bytes, drain)) return p;
    if (plain_cap_ >= bytes) return plain_;
    drain();
    std::free(plain_);
    plain_ = std::malloc(bytes);
    plain_cap_ = plain_ ? bytes : 0;
    return plain_;
  }

 private:
  Lock lock_;
  Unlock unlock_;
  std::size_t max_;
  int requests_ = 0;
  void *locked_ = nullptr, *plain_ = nullptr;
  std::size_t locked_cap_ = 0, plain_cap_ = 0;
};

// Waits for the copies in flight on every return but the one after done(): a call that fails half
// way through leaves none that would read the staging block, or write the device record, when the
// next call (on another stream, maybe) uses them again.
template <class Drain>
class DrainGuard {
 public:
  explicit DrainGuard(Drain drain) : drain_(drain) {}
  DrainGuard(const DrainGuard&) = delete;
  DrainGuard& operator=(const DrainGuard&) = delete;
  ~DrainGuard() {
    if (armed_) drain_();
  }
  void done() { armed_ = false; }

 private:
  Drain drain_;
  bool armed_ = true;
};

}  // namespace thor
