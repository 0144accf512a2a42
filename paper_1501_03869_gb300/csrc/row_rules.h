// row_rules.h -- rules by which launches choose kernels and shapes, in plain C++
// so that a host test can check them (internal).
#pragma once

#include <cstddef>
#include <cstdint>

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

// Shared-memory budget where `budget` is the one for short windows: that while its
// ring holds 32 / FB of the longest windows, else 110 KB while that holds two and a
// half, else the device's limit.  8 FP32 frames of 22 300 pixels x 512 sensors with
// windows of 320 / 632 / 1 248 rows: 87 / 130 us in 72 KB, 89 / 117 / 184 in 110
// KB, 120 / 133 / 184 in all; 4 frames with 632 / 1 248 rows: 79 / 120 us, 74 / 113,
// 81 / 112.  (For a class of a plan, `window` is the mean over its instances' units:
// one long record must not leave 32 uneven instances a CTA per SM, 3.80 ms against
// 2.67.)
inline size_t ring_budget(size_t budget, size_t fixed, size_t window, int FB, size_t limit) {
  const size_t two = size_t(110) * 1024;
  if (fixed + size_t(32 / FB) * window <= budget) return budget;
  if (budget < two && two <= limit) budget = two;
  return fixed + window * 5 / 2 <= budget ? budget : limit;
}

// Resident CTAs per SM of the windowed single-frame gather: what its registers
// allow (weights and computed delays hold more) and, for slots above 288 rows,
// its shared memory.
constexpr int window_ctas(bool delays, bool weights, int rows) {
  return delays || weights ? 6 : (rows > 288 ? 7 : 9);
}

// Whether a single frame goes through the windowed kernel; else the integrand is
// gathered from L2 by a kernel with 8 CTAs per SM or more.  Stored delays of up
// to 288 rows always do.  The other forms hold fewer CTAs, so a launch whose last
// wave is nearly empty loses what windows save: they need their share of a wave's
// (or, with more, of all waves') slots.  256 x 256 nodes, 512 sensors, GPU time
// windowed / from L2, by units over resident CTAs:
//   table, 289-384 rows  1.02: 20.0 / 16.9 us   1.31: 20.6 / 21.5   2.8: 30.5 / 38.5
//     256-pixel tiles    0.51: 20.5 / 18.2      0.62: 20.6 / 22.4   1.1: 35.9 / 31.2
//   table with weights   0.32: 15.9 / 15.4      0.88: 16.3 / 19.8   2.1: 37.3 / 34.8
//                        1.18: 26.3 / 24.1      1.53: 26.6 / 26.7   3.2: 50.3 / 54.5
//   constant speed       0.32: 15.0 / 13.9      1.82: 25.0 / 26.9   2.1: 34.0 / 30.9
//     129-192 rows       1.44: 28.2 / 23.6      0.88: 17.0 / 17.2   2.6: 39.6 / 35.6
//     with weights       0.32: 19.5 / 14.6      0.88: 20.1 / 22.5   2.6: 47.5 / 49.0
// With one segment per tile the windowed kernel saves the reduction's launch, which
// is worth more than that in one wave (64 sensors, constant speed 8.7 / 12.6 us,
// with weights 10.0 / 13.0).
inline bool window_pays(bool delays, bool weights, int P, int rows, int64_t units, int n_seg, int n_sm) {
  if (rows < 0 || rows > (delays ? 192 : (weights ? 288 : 384)) || (delays && P != 128)) return false;
  if (!delays && !weights && rows <= 288) return true;
  const int64_t wave = int64_t(window_ctas(delays, weights, rows)) * n_sm;
  const int64_t waves = (units + wave - 1) / wave;
  if (n_seg == 1 && waves == 1) return true;
  if (delays && !weights && rows > 128) return false;
  const int percent = delays ? 80 : (weights ? (waves == 1 ? 40 : 75) : (waves == 1 ? 60 : 65));
  return units * 100 >= percent * waves * wave;
}

}  // namespace patbp
