// launch_cache.h -- what a persistent kernel's launch asks the driver, kept per
// device.  Host code without CUDA types, so that it can be tested by itself.
#pragma once

#include <atomic>
#include <cstddef>

namespace bilu {

// Devices whose answers are kept; a launch on any other asks each time.
constexpr int kMaxCachedDevices = 64;

// The CTAs of one kernel that fit on an SM with a given amount of dynamic shared
// memory.  The answer, and the kernel's shared-memory limit that query() raises
// with it, belong to a device, and launches come from several threads: one word
// per device holds (bytes << 8) | CTAs of the last question, so no thread can
// pair one question with another's answer, and a thread that finds another size
// there asks again.  query(bytes) must leave the kernel launchable with ANY size
// (set the limit to the most there is, never to `bytes`: another thread may be
// about to launch with more).
class LaunchCache {
 public:
  template <typename Query>
  int ctas_per_sm(int device, size_t bytes, Query query) {
    if (device < 0 || device >= kMaxCachedDevices) return clamp(query(bytes));
    std::atomic<unsigned long long>& slot = slots_[device];
    const unsigned long long have = slot.load(std::memory_order_acquire);
    if ((have & 255u) != 0 && (have >> 8) == bytes) return (int)(have & 255u);
    const int ctas = clamp(query(bytes));
    slot.store(((unsigned long long)bytes << 8) | (unsigned long long)ctas, std::memory_order_release);
    return ctas;
  }

 private:
  static int clamp(int ctas) { return ctas < 1 ? 1 : ctas > 255 ? 255 : ctas; }
  std::atomic<unsigned long long> slots_[kMaxCachedDevices] = {};
};

}  // namespace bilu
