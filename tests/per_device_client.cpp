// The values of per_device.h on made-up devices: prints "ok" when each device
// is asked once, however many threads want it, and a failure is not kept.
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>

#include "per_device.h"

int main() {
  cpra::PerDevice<int> facts;
  std::atomic<int> asked[3] = {};
  std::atomic<bool> wrong{false};
  auto want = [&](int dev) {
    int v = -1;
    const int e = facts.get(dev, v, [&](int& t) {
      const int n = asked[dev]++;
      if (dev == 2 && n == 0) return 7;  // the first try on device 2 fails
      t = 100 + dev;
      return 0;
    });
    if (e == 0 ? v != 100 + dev : (e != 7 || v != -1)) wrong = true;
  };
  std::vector<std::thread> th;
  for (int i = 0; i < 8; ++i)
    th.emplace_back([&] {
      for (int k = 0; k < 300; ++k) want(k % 3);
    });
  for (auto& t : th) t.join();
  if (wrong || asked[0] != 1 || asked[1] != 1 || asked[2] != 2) return 1;
  std::puts("ok");
  return 0;
}
