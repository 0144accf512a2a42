// row_rules.h -- rules of the batched gather's launch shapes, in plain C++ so
// that a host test can check them (internal).
#pragma once

#include <cstddef>

namespace patbp {

// Below, `fixed` is what a CTA's shared memory holds besides the ring and
// `window` the bytes of the longest window.

// Whether rows of FB frames suit the windows: a ring of fewer than three of the
// longest windows copies and interpolates in turn, and rows of half the length
// are faster (32 FP32 frames of 8 700 pixels x 96 sensors, windows of 1 104 rows
// of 128 bytes: 113 us in rows of 32, 70 of 16; 16 frames with 2 192 rows: 108
// us in rows of 16, 72 of 8).  Rows of 4 give way below four windows, to single
// frames, whose copies are small (4 / 16 / 32 frames with 3 280 rows: 51 / 102 /
// 151 us in rows of 4, 37 / 94 / 149 alone; with 6 272 rows 85 / 188 / 281, 48 /
// 129 / 240).
inline bool ring_is_deep(int FB, size_t fixed, size_t window, size_t limit) {
  return fixed + (FB == 4 ? 4 : 3) * window <= limit;
}

// Shared-memory budget where `budget` is the one for short windows: the
// smallest of it, 110 KB and the device's limit whose ring holds 32 / FB of the
// longest windows.  8 FP32 frames of 22 300 pixels x 512 sensors with windows of
// 320 / 632 rows: 87 / 130 us in 72 KB, 89 / 117 in 110 KB, 120 / 133 in all; 4
// frames with 632 / 1 248 rows: 79 / 120 us, 74 / 113, 81 / 112.
inline size_t ring_budget(size_t budget, size_t fixed, size_t window, int FB, size_t limit) {
  const size_t need = fixed + size_t(32 / FB) * window;
  if (need <= budget) return budget;
  const size_t two = size_t(110) * 1024;
  return budget < two && two <= limit && need <= two ? two : limit;
}

}  // namespace patbp
