// row_rules.cpp -- test harness: the batched gather's rules for long windows.
// Built and run by tests/test_row_rules.py.
#include <cstdio>
#include <initializer_list>

#include "row_rules.h"

using namespace patbp;

int main() {
  int bad = 0;
  auto need = [&](bool ok, const char* what, int FB, size_t rows) {
    if (!ok && ++bad < 20) std::printf("%s: FB %d rows %zu\n", what, FB, rows);
  };
  const size_t limit = 227 * 1024, fixed = 9000;
  for (int FB : {4, 8, 16, 32}) {
    const size_t first = FB >= 16 ? limit : 72 * 1024;
    size_t last = 0;
    for (size_t rows = 8; rows < 9000; rows += 8) {
      const size_t window = rows * FB * 4;
      const size_t b = ring_budget(first, fixed, window, FB, limit);
      need(b == first || b == 110 * 1024 || b == limit, "an unknown budget", FB, rows);
      need(b >= last, "a smaller budget for longer windows", FB, rows);
      last = b;
      // the default until the ring gets shallow, and never more than needed
      if (fixed + 32 / FB * window <= first) need(b == first, "short windows leave the default", FB, rows);
      else need(b > first || first == limit, "long windows in the default budget", FB, rows);
      if (b < limit) need(fixed + 32 / FB * window <= b, "a shallow ring below the limit", FB, rows);
      // rows whose ring holds fewer than three windows give way (rows of 4: four)
      need(ring_is_deep(FB, fixed, window, limit) == ((limit - fixed) / window >= (FB == 4 ? 4u : 3u)), "deep", FB, rows);
    }
  }
  // what rows of 32 cannot hold, rows of 8 can
  need(!ring_is_deep(32, fixed, 1752 * 128, limit) && ring_is_deep(8, fixed, 1752 * 32, limit), "1 752 rows", 32, 1752);
  need(ring_budget(72 * 1024, fixed, 12000, 8, 100 * 1024) == 72 * 1024, "a device with less", 8, 0);
  need(ring_budget(72 * 1024, fixed, 22000, 8, 100 * 1024) == 100 * 1024, "a device with less than 110 KB", 8, 0);
  if (bad) return 1;
  std::printf("ok\n");
  return 0;
}
