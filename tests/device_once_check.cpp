// DeviceOnce: once per device, again after a failure, for any device number and
// from several threads.  Prints 1 for each that holds.
#include <cstdio>
#include <thread>
#include <vector>

#include "../paper_1305_2418_gb300/csrc/device_once.h"

int main() {
  DeviceOnce once;
  int n[70] = {};
  auto act = [&](int dev, int e) { return once(dev, [&] { ++n[dev]; return e; }); };
  for (int q = 0; q < 3; ++q) act(0, 0);
  for (int q = 0; q < 3; ++q) act(1, 0);  // another device of the same process
  const bool each = n[0] == 1 && n[1] == 1;
  const bool failed = act(2, 7) == 7 && act(2, 7) == 7 && act(2, 0) == 0 && act(2, 7) == 0;
  act(69, 0);
  act(69, 0);
  int none = 0;
  once(-1, [&] { ++none; return 0; });
  const bool beyond = n[69] == 2 && none == 1;
  DeviceOnce shared;
  std::atomic<int> done{0}, seen{0};
  std::vector<std::thread> t;
  for (int q = 0; q < 8; ++q)
    t.emplace_back([&] {
      for (int i = 0; i < 1000; ++i) {
        shared(i & 3, [&] { return done.fetch_or(1 << (i & 3)), 0; });
        seen += (done.load() >> (i & 3)) & 1;  // done before any call returns
      }
    });
  for (auto& q : t) q.join();
  std::printf("%d %d %d %d\n", each, failed && n[2] == 3, beyond, seen.load() == 8000);
  return 0;
}
