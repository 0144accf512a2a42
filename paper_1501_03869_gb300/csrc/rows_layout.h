// rows_layout.h -- shared memory of the batched gather (gather_rows.cuh), in
// plain C++ so that a host test can check it (internal).
//
// Header, then a ring of StreamParams::ring bytes that is filled with groups of
// up to S consecutive sensors (kSlots groups at most), then 2 zero rows that
// out-of-record pixels read, then the running sums of whole-tile units.  A
// group takes the bytes it needs: windows differ threefold between tiles and
// sensors, and fixed stages sized for the longest sum left two or three stages
// in flight.
//   u    [se][P] float    table rows, or [se][8] float anchors (constant speed)
//   wa   [se][8] float    solid-angle weight anchors (mode bit 1 only)
//   m    [se][FB] float   multipliers w_s * sigma
//   win  [rows][FB]       the windows back to back (128-byte aligned)
// Every byte of a group arrives by a bulk copy.  What warps write with
// ordinary stores (barriers, headers, records) has a fixed place in the header:
// groups start anywhere in the ring, so an ordinary store there could meet a
// later bulk copy to the same bytes, which the memory model orders only behind
// a proxy fence.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PATBP_HD __host__ __device__
#else
#define PATBP_HD
#endif

namespace patbp {

constexpr int kSlots = 8;
constexpr int kRowsMaxS = 16;  // sensors of a group
// A group of several sensors takes at most this part of the ring.  Fewer, larger
// groups win where rows are short (12 BF16 frames in rows of 8, 120 tiles: half the
// ring 33.3 us, a third 35.3; only 32 uneven instances would have it otherwise, 2.58
// and 2.54 ms), more groups in flight where they are long (12 and 32 frames of that
// series in rows of 16 and 32: half 0.7 and 1.2 % slower; a quarter loses in both).
PATBP_HD constexpr int rows_share(int FB) { return FB >= 16 ? 3 : 2; }
constexpr int kSegs = 10;      // segments alive: one per slot, one being planned, one spare

struct alignas(8) RowsRecord {  // one sensor of a group: window address and row limit (as bits)
  uint32_t window, limit;
};

struct alignas(8) RowsSensor {  // window base | length << 16, rows of the segment before it
  uint32_t base_len, before;
};

struct RowsSegment {           // what the copiers need of a (unit, segment)
  RowsSensor sensor[64];
  uint64_t u, wa, b, m;        // addresses of the segment's first sensor
  uint64_t stride;             // bytes from one sensor's integrand rows to the next's
  uint64_t pad;
};

// Header: barriers, unit ring, slot headers and the abort flag | window bases
// [2][64], the one part that bulk copies write | records | segments.
constexpr int kRowsMeta = 512;
constexpr int kRowsRecs = kRowsMeta + 2 * 64 * 4;
constexpr int kRowsSegs = kRowsRecs + kSlots * kRowsMaxS * int(sizeof(RowsRecord));
constexpr int kRowsHeader = (kRowsSegs + kSegs * int(sizeof(RowsSegment)) + 127) / 128 * 128;

struct RowsGroup {
  uint32_t wa, m, end, win;  // end: bytes copied before the windows
  PATBP_HD RowsGroup(int se, int P, int FB, int mode) {
    wa = (mode & 1) ? uint32_t(se) * 32u : uint32_t(se) * uint32_t(P) * 4u;
    m = wa + ((mode & 2) ? uint32_t(se) * 32u : 0u);
    end = m + uint32_t(se) * uint32_t(FB) * 4u;
    win = (end + 127u) & ~127u;
  }
  // bytes of the group's bulk copies
  PATBP_HD uint32_t copied(int rows, int FB) const { return end + uint32_t(rows) * uint32_t(FB) * 4u; }
  PATBP_HD uint32_t bytes(int rows, int FB) const {
    return (win + uint32_t(rows) * uint32_t(FB) * 4u + 127u) & ~127u;
  }
};

}  // namespace patbp
