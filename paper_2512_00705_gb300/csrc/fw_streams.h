// fw_streams.h -- how many streams a graph's walks are launched on (host code
// without CUDA, tested on the CPU).
#pragma once

#include <chrono>
#include <cstdint>
#include <mutex>

namespace fw {

// Callers that walk on several streams at once cannot say so in a call, but
// their launches alternate between streams.  note() counts the streams used
// within the last kWindow, this launch's included: an estimate of the launches
// in flight, for the choice of a launch shape only (rows never depend on it).
// A launch takes 0.02 to a few ms; a stream not used for longer than kWindow
// is idle or holds one launch that fills the GPU in any shape.  Stream handles
// are compared, never used.
class RecentStreams {
 public:
  using Clock = std::chrono::steady_clock;
  static constexpr std::chrono::milliseconds kWindow{10};
  static constexpr int kMost = 16;  // streams told apart

  int note(uintptr_t stream, Clock::time_point now = Clock::now()) {
    std::lock_guard<std::mutex> lk(mu_);
    int active = 1, mine = -1, oldest = 0;
    for (int i = 0; i < used_; ++i) {
      if (seen_[i].stream == stream) mine = i;
      else if (now - seen_[i].at <= kWindow) ++active;
      if (seen_[i].at < seen_[oldest].at) oldest = i;
    }
    if (mine < 0) mine = used_ < kMost ? used_++ : oldest;
    seen_[mine] = {stream, now};
    return active < kMost ? active : kMost;
  }

 private:
  struct Seen {
    uintptr_t stream;
    Clock::time_point at;
  };
  std::mutex mu_;
  Seen seen_[kMost] = {};
  int used_ = 0;
};

}  // namespace fw
