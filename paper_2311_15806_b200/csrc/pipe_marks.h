// Which streams have an expansion as their last library call (host logic only, no CUDA).
#pragma once

#include <atomic>
#include <cstdint>
#include <mutex>

namespace pipe {

// A stream as the table tells streams apart: the handle alone does not, for the default stream has the same one on every device,
// two of them (null and 1, cudaStreamLegacy) on each, and the per-thread default stream (2) the same one in every thread.  (Asking the runtime for a
// stream's id would settle all of this, but invalidates a capture that the stream is in.)
struct StreamKey {
  int device = -1;      // -1: the runtime did not say which device is current
  uint64_t handle = 0;
  uint64_t thread = 0;  // of the per-thread default stream
  bool known() const { return device >= 0; }
  bool operator==(const StreamKey& o) const { return device == o.device && handle == o.handle && thread == o.thread; }
};
inline StreamKey stream_key(int device, uint64_t handle) {
  constexpr uint64_t kLegacy = 1, kPerThread = 2;
  static std::atomic<uint64_t> threads{0};
  StreamKey k;
  k.device = device;
  k.handle = handle ? handle : kLegacy;
  if (handle == kPerThread) {
    thread_local const uint64_t id = ++threads;
    k.thread = id;
  }
  return k;
}

// The marks of one process.  Calls that name a stream the table cannot tell from others, and every call once there were more
// marked streams than the table holds, are answered as if an expansion stood before them: that costs a wait, never a result.
class ExpansionMarks {
 public:
  static constexpr int kMax = 64;
  // (no mark anywhere: the usual case, decided without a lock)
  bool none() const { return count_.load(std::memory_order_acquire) == 0; }
  void mark(const StreamKey& s) {
    std::lock_guard<std::mutex> lock(mu_);
    if (s.known())
      for (int i = 0; i < n_; ++i)
        if (marked_[i] == s) return;
    if (s.known() && n_ < kMax) marked_[n_++] = s;
    else always_ = true;
    count_.store(n_ + (always_ ? 1 : 0), std::memory_order_release);
  }
  bool marked(const StreamKey& s) {
    std::lock_guard<std::mutex> lock(mu_);
    return find(s) != kNone;
  }
  bool take(const StreamKey& s) {
    std::lock_guard<std::mutex> lock(mu_);
    const int i = find(s);
    if (i >= 0) {
      marked_[i] = marked_[--n_];
      count_.store(n_ + (always_ ? 1 : 0), std::memory_order_release);
    }
    return i != kNone;
  }

 private:
  static constexpr int kNone = -1, kCannotTell = -2;
  int find(const StreamKey& s) const {
    if (s.known())
      for (int i = 0; i < n_; ++i)
        if (marked_[i] == s) return i;
    return always_ || (!s.known() && n_ > 0) ? kCannotTell : kNone;
  }
  std::mutex mu_;
  std::atomic<int> count_{0};
  StreamKey marked_[kMax];
  int n_ = 0;
  bool always_ = false;
};

}  // namespace pipe
