// rows_layout.cpp -- test harness: the shared-memory layout of the batched
// gather.  A group's place in the ring is filled by bulk copies alone (no
// ordinary store may share bytes with them: the memory model orders the two
// only behind a proxy fence), and what warps store has its own place in the
// header.  Built and run by tests/test_rows_layout.py.
#include <cstdio>
#include <initializer_list>

#include "rows_layout.h"

using namespace patbp;

int main() {
  int bad = 0;
  auto need = [&](bool ok, const char* what, int se, int P, int FB, int mode) {
    if (ok) return;
    if (++bad < 20) std::printf("%s: se %d P %d FB %d mode %d\n", what, se, P, FB, mode);
  };
  for (int P : {128, 256})
    for (int FB : {4, 8, 16, 32})
      for (int mode = 0; mode < 4; ++mode)
        for (int se = 1; se <= kRowsMaxS; ++se)
          for (int rows : {0, 8, 120, 1752}) {
            const RowsGroup L(se, P, FB, mode);
            // the copies in order: delay data, weight anchors, multipliers, windows
            const uint32_t u = (mode & 1) ? se * 32u : se * P * 4u;
            const uint32_t wa = (mode & 2) ? se * 32u : 0u, m = se * FB * 4u, win = rows * FB * 4u;
            need(L.wa == u && L.m == u + wa && L.end == u + wa + m, "a gap between copies", se, P, FB, mode);
            need(L.win >= L.end && L.win - L.end < 128 && L.win % 128 == 0, "padding before the windows", se, P, FB, mode);
            need(L.copied(rows, FB) == u + wa + m + win, "bytes a group waits for", se, P, FB, mode);
            need(L.bytes(rows, FB) >= L.win + win && L.bytes(rows, FB) - L.win - win < 128 &&
                     L.bytes(rows, FB) % 128 == 0,
                 "bytes of a group", se, P, FB, mode);
            need(L.wa % 16 == 0 && L.m % 16 == 0, "copies start on 16 bytes", se, P, FB, mode);
          }
  // header parts one after the other, all before the ring
  need(kRowsMeta >= 8 * (3 * kSlots + 2) + 8 * 16 + 16 * kSlots + 4, "barriers, rings, slot headers", 0, 0, 0, 0);
  need(kRowsRecs - kRowsMeta == 2 * 64 * 4 && kRowsMeta % 16 == 0, "window bases", 0, 0, 0, 0);
  need(sizeof(RowsRecord) == 8 && kRowsSegs - kRowsRecs == kSlots * kRowsMaxS * 8 && kRowsRecs % 8 == 0, "records", 0, 0, 0, 0);
  need(kRowsHeader >= kRowsSegs + kSegs * int(sizeof(RowsSegment)) && kRowsSegs % 8 == 0, "segments", 0, 0, 0, 0);
  need(kRowsHeader % 128 == 0, "the ring starts on 128 bytes", 0, 0, 0, 0);
  if (bad) return 1;
  std::printf("ok\n");
  return 0;
}
