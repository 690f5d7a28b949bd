// Host test of LaunchCache: eight threads ask for different sizes on different
// devices at once; every answer must be the one of its own (device, size), and
// the pretended per-device limit must hold whatever a thread launches with.
#include <cstdio>
#include <thread>
#include <vector>

#include "launch_cache.h"

int main() {
  bilu::LaunchCache cache;
  constexpr int kDevices = bilu::kMaxCachedDevices + 2;
  std::vector<std::atomic<int>> limit(kDevices), asked(kDevices);
  std::atomic<int> wrong{0};
  auto answer = [](int dev, size_t bytes) { return 1 + (int)((dev * 31 + bytes / 1024) % 20); };
  auto worker = [&](int t) {
    for (int it = 0; it < 20000; ++it) {
      const int dev = (it * 7 + t) % kDevices;
      const size_t bytes = 1024 * (size_t)(1 + (it / 3 + t) % 4);
      const int got = cache.ctas_per_sm(dev, bytes, [&](size_t b) {
        limit[dev] = 227 * 1024;
        asked[dev]++;
        return answer(dev, b);
      });
      if (got != answer(dev, bytes) || limit[dev] < (int)bytes) wrong++;
    }
  };
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t) ts.emplace_back(worker, t);
  for (auto& t : ts) t.join();
  // one size on one device: asked once, on another device again
  bilu::LaunchCache one;
  int n0 = 0, n1 = 0;
  for (int q = 0; q < 5; ++q) one.ctas_per_sm(0, 64, [&](size_t) { ++n0; return 3; });
  for (int q = 0; q < 5; ++q) one.ctas_per_sm(1, 64, [&](size_t) { ++n1; return 5; });
  const bool none = one.ctas_per_sm(2, 64, [](size_t) { return 0; }) == 1;  // never less than one
  std::printf("wrong %d, asked %d %d\n", wrong.load(), n0, n1);
  return wrong == 0 && n0 == 1 && n1 == 1 && none ? 0 : 1;
}
