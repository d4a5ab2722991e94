// How many calls are at work on a device, for the launch geometry of the kernels
// that stay resident for a whole level (host code).
//
// Such a kernel fills an SM with a block, and a cooperative launch of the whole
// chip waits until every other one has left it; calls that run at the same time
// (handles of several host threads, the executor's jobs) therefore take at most
// half the chip each, and a call that is alone takes all of it.  The count is only
// a measure of the load: results do not depend on it, and a launch that was sized
// before another call came is over within its level.
#pragma once

#include <atomic>

namespace hgk {

constexpr int IN_FLIGHT_DEVICES = 64;

inline std::atomic<int>& calls_in_flight(int device) {
  static std::atomic<int> count[IN_FLIGHT_DEVICES];
  return count[(unsigned)device % IN_FLIGHT_DEVICES];
}

// Counts one call while it lives.  `depth`: of the handle, whose calls nest
// (hg_partition makes others) and count once.
class CallScope {
 public:
  CallScope(int device, int& depth) : count_(calls_in_flight(device)), depth_(depth) {
    if (depth_++ == 0) count_.fetch_add(1, std::memory_order_relaxed);
  }
  ~CallScope() {
    if (--depth_ == 0) count_.fetch_sub(1, std::memory_order_relaxed);
  }
  CallScope(const CallScope&) = delete;
  CallScope& operator=(const CallScope&) = delete;

 private:
  std::atomic<int>& count_;
  int& depth_;
};

}  // namespace hgk
