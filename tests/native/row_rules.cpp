// row_rules.cpp -- test harness: the batched gather's rules for long windows and
// the single-frame gather's choice of kernel.
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
      if (b < limit) need(fixed + 5 * window / 2 <= b, "a shallow ring below the limit", FB, rows);
      // rows whose ring holds fewer than three windows give way (rows of 4: four)
      need(ring_is_deep(FB, fixed, window, limit) == ((limit - fixed) / window >= (FB == 4 ? 4u : 3u)), "deep", FB, rows);
    }
  }
  // what rows of 32 cannot hold, rows of 8 can
  need(!ring_is_deep(32, fixed, 1752 * 128, limit) && ring_is_deep(8, fixed, 1752 * 32, limit), "1 752 rows", 32, 1752);
  need(ring_budget(72 * 1024, fixed, 12000, 8, 100 * 1024) == 72 * 1024, "a device with less", 8, 0);
  need(ring_budget(72 * 1024, fixed, 40000, 8, 100 * 1024) == 100 * 1024, "a device with less than 110 KB", 8, 0);
  need(ring_budget(110 * 1024, fixed, 30000, 8, limit) == 110 * 1024 && ring_budget(110 * 1024, fixed, 45000, 8, limit) == limit,
       "from 110 KB", 8, 0);
  const int n_sm = 152;
  auto pays = [&](bool delays, bool weights, int P, int rows, int64_t units, int n_seg) {
    return window_pays(delays, weights, P, rows, units, n_seg, n_sm);
  };
  for (int P : {128, 256})
    for (int64_t units : {int64_t(1), int64_t(900), int64_t(1400), int64_t(9000), int64_t(500000)})
      for (int n_seg : {1, 8}) {
        // stored delays without weights: every slot up to 288 rows
        need(pays(false, false, P, 288, units, n_seg), "288 rows", P, units);
        need(!pays(false, false, P, 385, units, n_seg) && !pays(false, true, P, 289, units, n_seg) &&
                 !pays(true, false, P, 193, units, n_seg) && !pays(true, true, P, 193, units, n_seg),
             "no slot holds these", P, units);
        need(!pays(true, false, 256, 64, units, n_seg), "constant speed has no 256-pixel form", P, units);
        // many waves: the last one does not matter
        if (units == 500000) {
          need(pays(false, false, P, 384, units, n_seg) && pays(false, true, P, 288, units, n_seg), "volumes", P, units);
          need(pays(true, false, 128, 128, units, n_seg) && !pays(true, false, 128, 136, units, n_seg) &&
                   pays(true, true, 128, 192, units, n_seg),
               "volumes at constant speed", P, units);
        }
      }
  // one segment per tile and one wave: no reduction
  need(pays(true, false, 128, 192, 48, 1) && pays(true, true, 128, 64, 48, 1) && pays(false, true, 256, 64, 48, 1) &&
           pays(false, false, 128, 384, 48, 1),
       "one segment", 0, 48);
  // launches that ran slower than from L2 (the table in row_rules.h)
  need(!pays(false, false, 128, 296, 1080, 8) && !pays(false, false, 256, 360, 544, 8) &&
           !pays(false, false, 256, 344, 1184, 8),
       "a table's 384-row slots", 0, 0);
  need(!pays(false, true, 128, 80, 288, 8) && !pays(false, true, 128, 88, 1080, 8) && !pays(false, true, 128, 96, 1944, 8),
       "weights", 0, 0);
  need(!pays(true, false, 128, 96, 288, 8) && !pays(true, false, 128, 120, 1944, 8) && !pays(true, false, 128, 168, 1312, 8) &&
           !pays(true, false, 128, 176, 2368, 8) && !pays(true, true, 128, 96, 288, 8) && !pays(true, true, 128, 96, 1312, 8),
       "constant speed", 0, 0);
  // and ones that ran faster
  need(pays(false, false, 128, 312, 1392, 8) && pays(false, false, 256, 360, 696, 8) && pays(false, true, 256, 248, 656, 8) &&
           pays(false, true, 128, 88, 800, 8) && pays(false, true, 128, 104, 2944, 8) && pays(true, false, 128, 104, 1656, 8) &&
           pays(true, true, 128, 136, 800, 8),
       "windows that pay", 0, 0);
  if (bad) return 1;
  std::printf("ok\n");
  return 0;
}
