// smem_grant.cpp -- test harness: shared-memory grants against a fake of the
// attribute call.  Every device gets its own, a refused call grants nothing,
// and no launch ever finds less than it asked for, whatever other threads ask.
// Built and run by tests/test_smem_grant.py.
#include <atomic>
#include <cstdio>
#include <random>
#include <thread>
#include <vector>

#include "smem_grant.h"

int main() {
  std::atomic<size_t> attr[4] = {};
  std::atomic<int> bad{0};
  {
    patbp::SmemGrant g;
    auto set = [&](int dev) {
      return [&, dev](size_t b) {
        attr[dev] = b;
        return 0;
      };
    };
    g.ensure(0, 100, set(0));
    g.ensure(1, 80, set(1));
    if (attr[0] != 100 || attr[1] != 80) bad += 1;  // the second device has its own grant
    g.ensure(0, 60, set(0));
    if (attr[0] != 100) bad += 1;  // never less
    if (g.ensure(0, 200, [](size_t) { return 7; }) != 7) bad += 1;
    g.ensure(0, 200, set(0));
    if (attr[0] != 200) bad += 1;  // a refused call is made again
    if (g.ensure(1000, 10, [](size_t) { return 5; }) != 5) bad += 1;
  }
  for (auto& a : attr) a = 0;
  patbp::SmemGrant g;
  std::vector<std::thread> pool;
  for (int t = 0; t < 8; ++t)
    pool.emplace_back([&, t] {
      std::mt19937 rng(t);
      for (int i = 0; i < 20000; ++i) {
        const int dev = int(rng() & 3);
        const size_t want = 1 + i + rng() % 4096;
        g.ensure(dev, want, [&](size_t b) {
          std::this_thread::yield();
          attr[dev] = b;
          return 0;
        });
        if (attr[dev] < want) bad += 1;
      }
    });
  for (auto& t : pool) t.join();
  if (bad) {
    std::printf("%d faults\n", int(bad));
    return 1;
  }
  std::printf("ok\n");
  return 0;
}
