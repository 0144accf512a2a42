// gather_rows.cuh -- the batched gather of Eq. (BP) for 4, 8, 16 or 32 frames
// per unit (internal).
//
//   out[f][r] = sum_s w_s * b_{f,s}(T_s(r)/dt) with linear interpolation.
//
// What bounds it: shared-memory wavefronts for FP32, instruction latency for
// 16-bit integrands.  Every (pixel, sensor) reads its integrand row (two rows
// for FP32) of FB frames from a window in shared memory.  The frames of a row
// lie across the lanes: a lane owns 4 or 8 frames of its pixels, so one
// 16-byte load per lane brings several whole rows.  A row of 32 frames fills
// the 32 banks and its loads never conflict.  Shorter rows share the banks;
// FP32 reads two consecutive rows anyway, one even and one odd, and half of
// the pixels of every quarter warp read the even one first, the other half the
// odd one, which makes 16-frame rows free of conflicts and lowers the 8-frame
// ones (lanes that own all 8 frames of a pixel, the mapping before this one,
// meet 1.82 wavefronts per load on the paper-shaped frame, 2.17 on a volume;
// this one 1.57 and 1.62, counted from the tables' rows).  Index arithmetic
// and FP32 arithmetic are packed or shared by the frames of a lane.
// Measured, whole calls (preprocessing and reduction included): 64 FP32 frames
// of 512 sensors x 21 323 pixels 489 -> 317 us; 8 BF16 frames of 640 sensors x
// 1.04 M voxels 3.16 -> 2.14 ms; 64 BF16 frames of 64 x 6 092 54 -> 33 us; 12
// FP16 frames with solid-angle weights 166 -> 127 us.
//
// Work: one unit is (frame group, tile) with all segments of G sensors when
// there are many units, else (frame group, tile, segment), whose sums
// rows_reduce_kernel adds in segment order.  A producer warp streams groups of
// at most S sensors (delay data, multipliers and windows) into a ring in
// shared memory with 1-D bulk copies completing on mbarriers.  The other warps own disjoint
// pixels and take every sensor, in order, so no sums are exchanged between
// warps: the sensor phases (s - s_lo) mod SW have an accumulator each, added
// in phase order at the end of a segment.  Per pixel the additions are those
// of gather_kernel and of the single-frame kernels (phases in order inside a
// segment, segments in order): a frame has the same bits alone and in a batch.
//
// As in gather.cuh the kernel is a programmatic dependent of the
// preprocessing: plain global loads use ld.global.cg, and every wait on an
// mbarrier is bounded.
#pragma once

#include "gather.cuh"
#include "packed.cuh"
#include "rows_layout.h"

namespace patbp {

// ------------------------------------------------------------------ shape --
template <int P, int FB, int FMT, int MODE>
struct RowsShape {
  // 16-byte quads of a row that a lane owns: two where the two loads can be
  // kept free of bank conflicts (halves the index work per update), and in
  // 8-frame rows where offsets or weights are computed, whose arithmetic then
  // stays in one lane without shuffles (24 FP32 frames of 22 300 pixels x 512
  // sensors, constant speed with weights: 294 -> 259 us, 256-pixel tiles 263 ->
  // 222; stored delays are faster with one, 198 us against 201).
  static constexpr int NQ = FB == 32 || (FB == 16 && FMT == kBF32) || (FB == 8 && MODE != 0) ? 2 : 1;
  static constexpr int LPP = FB / (4 * NQ);               // lanes that share a pixel
  static constexpr int PPW = 32 / LPP;                    // pixels of one warp-wide load
  static constexpr int NW = FB >= 16 ? 8 : 4;             // consumer warps
  static constexpr int NC = FB >= 16 ? 2 : 1;             // copier warps
  static constexpr int NPX = P / NW;                      // pixels of a warp
  static constexpr int A = NPX / PPW;                     // pixels of a lane
  static constexpr int V = A < 4 ? A : (NQ == 2 ? 4 : 2); // of which neighbours in the tile
  static constexpr int THREADS = 32 * (NW + 1 + NC);
  // resident CTAs per SM the registers must allow: 11 to 18 warps.  8-frame rows
  // spill in the 96 registers of three where a lane computes offsets or weights:
  // two are faster there (24 FP32 frames as above, constant speed, 256-pixel tiles
  // 234 -> 204 us; 12 frames of 6 600 pixels x 128 sensors 34 -> 28 us, with weights
  // too 39 -> 31).  With a table one call of 24 frames gains as well (184 -> 166),
  // but 32 uneven instances lose (2.62 -> 2.81 ms).
  static constexpr int MIN_CTAS = FB >= 16 ? 1 : (FB == 8 && MODE != 0 ? 2 : 3);
  static_assert(A % V == 0 && NPX * NW == P, "pixels of a lane");
};

struct RowsUnit {
  int inst, fg, tile, seg0, seg1;
};

// Units run segment by segment (split), then tile by tile with the frame
// groups of a tile next to each other: they share its table block in L2, and
// the integrand rows in use at a time are those of one segment.
__device__ __forceinline__ RowsUnit decode_rows(const StreamParams& p, int64_t u, int& inst) {
  while (inst + 1 < p.n_inst && u >= p.inst[inst + 1].unit_begin) ++inst;
  const InstDesc& d = p.inst[inst];
  const int64_t loc = u - d.unit_begin, per_seg = int64_t(d.n_tiles) * d.n_fg;
  RowsUnit q;
  q.inst = inst;
  q.seg0 = p.split ? int(loc / per_seg) : 0;
  q.seg1 = p.split ? q.seg0 + 1 : d.n_seg;
  const int64_t r = loc - q.seg0 * per_seg;
  q.tile = int(r / d.n_fg);
  q.fg = int(r - int64_t(q.tile) * d.n_fg);
  return q;
}

template <int P, int FB, int FMT, int SW, int MODE>
__global__ void __launch_bounds__(RowsShape<P, FB, FMT, MODE>::THREADS, RowsShape<P, FB, FMT, MODE>::MIN_CTAS)
    gather_rows_kernel(const __grid_constant__ StreamParams p) {
  using SH = RowsShape<P, FB, FMT, MODE>;
  constexpr int DELAYS = MODE & 1, WGT = (MODE >> 1) & 1;
  constexpr int A = SH::A, V = SH::V, NQ = SH::NQ, LPP = SH::LPP, PPW = SH::PPW, NPX = SH::NPX, NW = SH::NW;
  constexpr int NC = SH::NC;
  constexpr uint32_t ROW = FB * 4;               // bytes of one row
  constexpr uint32_t kMagic = 0x4B000000u;       // bit pattern of 2^23
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty = full + kSlots;
  uint64_t* plan_bar = empty + kSlots;
  uint64_t* meta_bar = plan_bar + kSlots;
  int64_t* unit_ring = reinterpret_cast<int64_t*>(meta_bar + 2);  // [kRing]
  uint4* slot_hdr = reinterpret_cast<uint4*>(unit_ring + kRing);  // [kSlots] (ring offset, sensors, first
                                                                  // sensor | segment << 16, rows)
  volatile int* abort_flag = reinterpret_cast<volatile int*>(slot_hdr + kSlots);
  uint32_t* meta = reinterpret_cast<uint32_t*>(smem + kRowsMeta);  // [2][64] packed bases
  RowsRecord* recs = reinterpret_cast<RowsRecord*>(smem + kRowsRecs);  // [kSlots][kRowsMaxS]
  RowsSegment* segs = reinterpret_cast<RowsSegment*>(smem + kRowsSegs);
  unsigned char* ring = smem + kRowsHeader;
  float* total = reinterpret_cast<float*>(ring + p.ring + 2 * ROW);  // [P][FB], whole-tile units
  const uint32_t ring_s = smem_addr(ring);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t N = p.n_units;

  if (threadIdx.x == 0) {
    for (int st = 0; st < kSlots; ++st) {
      mbar_init(&full[st], 2);  // planner and copier
      mbar_init(&empty[st], NW);
      mbar_init(&plan_bar[st], 1);
    }
    mbar_init(&meta_bar[0], 1);
    mbar_init(&meta_bar[1], 1);
    *abort_flag = 0;
    mbar_init_fence();
  }
  for (int q = threadIdx.x; q < 2 * FB; q += blockDim.x)
    reinterpret_cast<uint32_t*>(ring + p.ring)[q] = 0u;
  __syncthreads();

  if (warp > NW) {
    // ------------------------------------------------------------- copiers --
    // Copier c issues the copies of the groups in slots c, c + NC, ...: a lane
    // per window, one each for delay data, multipliers and weight anchors.  A
    // bulk copy costs its warp about 50 cycles to issue, so planning and
    // copying overlap in different warps (one producer warp for both took
    // 2000 cycles per group of 4 sensors and bounded the kernel).
    int slot = warp - NW - 1;
    uint32_t parity = 0;
    bool waited = false;
    for (;;) {
      if (!mbar_wait_bounded(&plan_bar[slot], parity, p.timeout_ns, abort_flag)) {
        if (lane == 0) {
          atomicOr(p.status, kStatusTimeout);
          *abort_flag = 1;
        }
        break;
      }
      const uint4 hdr = slot_hdr[slot];
      const int se = int(hdr.y), i0 = int(hdr.z & 0xffffu);
      if (se == 0) {  // end of work
        if (lane == 0) mbar_arrive(&full[slot]);
        break;
      }
      const RowsGroup L(se, P, FB, MODE);
      const RowsSegment& sg = segs[hdr.z >> 16];
      uint64_t src = 0;
      uint32_t dst = 0, bytes = 0;
      if (lane < se) {
        const RowsSensor x = sg.sensor[i0 + lane];
        const bool bad = hdr.w == 0xffffffffu;  // no room for the windows (a configuration error)
        const uint32_t w = bad ? uint32_t(p.ring) : hdr.x + L.win + (x.before - sg.sensor[i0].before) * ROW;
        // row r of the sensor's window is at rec.x + ROW * (2^23's bits + r);
        // the zero rows follow the ring
        recs[slot * kRowsMaxS + lane] =
            RowsRecord{ring_s + w - kMagic * ROW, __float_as_uint(float((uint32_t(p.ring) - w) / ROW))};
        src = sg.b + uint64_t(i0 + lane) * sg.stride + uint64_t((x.base_len & 0xffffu) * ROW);
        dst = ring_s + w;
        bytes = bad ? 0u : (x.base_len >> 16) * ROW;
      } else if (lane == 16) {
        src = sg.u + uint64_t(i0) * (DELAYS ? 32u : P * 4u);
        dst = ring_s + hdr.x;
        bytes = L.wa;
      } else if (WGT && lane == 17) {
        src = sg.wa + uint64_t(i0) * 32u;
        dst = ring_s + hdr.x + L.wa;
        bytes = L.m - L.wa;
      } else if (lane == 18) {
        src = sg.m + uint64_t(i0) * ROW;
        dst = ring_s + hdr.x + L.m;
        bytes = uint32_t(se) * ROW;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[slot]);  // the records are written
      const uint32_t bar = smem_addr(&full[slot]);
      auto copy = [&]() {
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
            "l"(src), "r"(bytes), "r"(bar)
            : "memory");
      };
      // delay data streams while the preprocessing grid still runs; its
      // outputs only after the wait
      const bool early = lane == 16 || lane == 17;
      if (!waited) {
        if (early && bytes) copy();
        __syncwarp();
        asm volatile("griddepcontrol.wait;" ::: "memory");
      }
      if (bytes && (waited || !early)) copy();
      waited = true;
      __syncwarp();
      slot += NC;
      if (slot >= kSlots) {
        slot -= kSlots;
        parity ^= 1u;
      }
    }
    if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
  } else if (warp == NW) {
    // ------------------------------------------------------------- planner --
    int inst = 0, inst_next = 0;
    // Slots in flight: `oldest` .. next - 1 (mod kSlots), n_fly of them, released
    // in order; `parity` is that of the oldest slot's use (it flips when
    // `oldest` wraps).  Ring space is counted in running byte totals (heads
    // and tails only grow; lane k keeps the total at the end of slot k's
    // group); `pos` is the head's place in the ring.
    int oldest = 0, next = 0, n_fly = 0;
    uint32_t parity = 0, head = 0, tail = 0, pos = 0, end_of = 0;
    const uint32_t ring_bytes = uint32_t(p.ring);
    auto abort_now = [&]() {
      if (lane == 0) {
        atomicOr(p.status, kStatusTimeout);
        *abort_flag = 1;
      }
    };
    auto seg_end = [&](const InstDesc& d, int seg) { return min(d.n_sensors, (seg + 1) * d.G); };
    // window bases of one (tile, segment) into meta slot `slot`
    auto issue_meta = [&](const InstDesc& d, int tile, int seg, int slot) {
      const int s_lo = seg * d.G;
      const uint32_t n4 = uint32_t((seg_end(d, seg) - s_lo + 3) & ~3);
      if (lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive_expect_tx(&meta_bar[slot], n4 * 4);
        bulk_g2s(meta + slot * 64, d.base + int64_t(tile) * d.n_sensors_pad + s_lo, n4 * 4,
                 &meta_bar[slot]);
      }
    };
    auto release_oldest = [&]() -> bool {
      if (!mbar_wait_bounded(&empty[oldest], parity, p.timeout_ns, abort_flag)) {
        abort_now();
        return false;
      }
      tail = __shfl_sync(0xffffffffu, end_of, oldest);
      if (++oldest == kSlots) {
        oldest = 0;
        parity ^= 1u;
      }
      --n_fly;
      return true;
    };
    // Publishes the group of `se` sensors from i0 of segment record `sg` in the
    // next slot, once the ring has `bytes` in one piece.
    auto publish = [&](int se, int i0, int sg, uint32_t rows) -> bool {
      const RowsGroup L(se, P, FB, MODE);
      uint32_t bytes = L.bytes(int(rows), FB);
      const bool bad = bytes > ring_bytes;  // cannot happen with a host-checked shape; stay in bounds
      if (bad) {
        rows = 0;
        bytes = L.bytes(0, FB);
      }
      uint32_t skip;
      for (;;) {
        if (n_fly == 0) pos = 0;
        skip = pos + bytes > ring_bytes ? ring_bytes - pos : 0u;
        if (n_fly == 0 || (n_fly < kSlots && head + skip + bytes - tail <= ring_bytes)) break;
        if (!release_oldest()) return false;
      }
      if (n_fly == 0) tail = head;
      const uint32_t at = skip ? 0u : pos;
      head += skip + bytes;
      pos = at + bytes;
      if (pos == ring_bytes) pos = 0;  // the next group starts at the front, with nothing skipped
      if (lane == next) end_of = head;
      if (lane == 0) {
        slot_hdr[next] = make_uint4(at, uint32_t(se), uint32_t(i0) | uint32_t(sg) << 16, bad ? 0xffffffffu : rows);
        if (bad) atomicOr(p.status, kStatusBadConfig);
        mbar_arrive_expect_tx(&full[next], L.copied(int(rows), FB));
        mbar_arrive(&plan_bar[next]);
      }
      ++n_fly;
      if (++next == kSlots) next = 0;
      return true;
    };
    // the first unit of every CTA is blockIdx.x; later ones come from the ticket
    auto next_ticket = [&]() -> int64_t {
      int64_t t = N;
      if (lane == 0)
        t = int64_t(gridDim.x) + int64_t(atomicAdd(reinterpret_cast<unsigned long long*>(p.sched), 1ull));
      return t;
    };
    int64_t t_cur = int64_t(blockIdx.x) < N ? int64_t(blockIdx.x) : N;
    int64_t t_next = t_cur < N ? next_ticket() : N;
    t_next = __shfl_sync(0xffffffffu, t_next, 0);
    if (t_next > N) t_next = N;
    int64_t j = 0;           // (unit, segment) items begun
    int64_t meta_last = -1;  // item of the last base copy requested
    if (t_cur < N) {
      const RowsUnit q = decode_rows(p, t_cur, inst);
      issue_meta(p.inst[q.inst], q.tile, q.seg0, 0);
      meta_last = 0;
    }
    // lane k: window rows that a group of k + 1 sensors may have
    const int room = int(ring_bytes / rows_share(FB) & ~127u) - int(RowsGroup(lane + 1, P, FB, MODE).win);
    const int cap = lane < p.S && room >= 0 ? room / (FB * 4) : -1;
    bool ok = true;
    int64_t ju = 0;
    int sgi = 0;  // next segment record
    for (; t_cur < N && ok; ++ju) {
      const RowsUnit q = decode_rows(p, t_cur, inst);
      const InstDesc& d = p.inst[q.inst];
      const int64_t t_next2 = t_next < N ? next_ticket() : N;
      if (lane == 0) unit_ring[ju % kRing] = t_cur;
      for (int seg = q.seg0; seg < q.seg1 && ok; ++seg, ++j) {
        const int slot = int(j & 1);
        if (!mbar_wait_bounded(&meta_bar[slot], uint32_t((j >> 1) & 1), p.timeout_ns, abort_flag)) {
          abort_now();
          ok = false;
          break;
        }
        __syncwarp();
        if (seg + 1 < q.seg1) {
          issue_meta(d, q.tile, seg + 1, slot ^ 1);
          meta_last = j + 1;
        } else if (t_next < N) {
          inst_next = inst;
          const RowsUnit qn = decode_rows(p, t_next, inst_next);
          issue_meta(p.inst[qn.inst], qn.tile, qn.seg0, slot ^ 1);
          meta_last = j + 1;
        }
        const int s_lo = seg * d.G, n = seg_end(d, seg) - s_lo;
        // the segment's record: windows and their running row counts, two
        // sensors per lane, and the addresses of its first sensor
        const uint32_t* mrow = meta + slot * 64;
        const uint32_t w0 = lane < n ? mrow[lane] : 0u, w1 = lane + 32 < n ? mrow[lane + 32] : 0u;
        uint32_t a0 = w0 >> 16, a1 = w1 >> 16;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t x = __shfl_up_sync(0xffffffffu, a0, o), y = __shfl_up_sync(0xffffffffu, a1, o);
          if (lane >= o) {
            a0 += x;
            a1 += y;
          }
        }
        a1 += __shfl_sync(0xffffffffu, a0, 31);
        RowsSegment& sg = segs[sgi];
        sg.sensor[lane] = RowsSensor{w0, a0 - (w0 >> 16)};
        sg.sensor[lane + 32] = RowsSensor{w1, a1 - (w1 >> 16)};
        if (lane == 0) {
          sg.u = DELAYS ? reinterpret_cast<uint64_t>(d.anchor + (int64_t(q.tile) * d.n_sensors_pad + s_lo) * 8)
                        : reinterpret_cast<uint64_t>(d.u + (int64_t(q.tile) * d.n_sensors + s_lo) * P);
          sg.wa = WGT ? reinterpret_cast<uint64_t>(d.wanchor + (int64_t(q.tile) * d.n_sensors_pad + s_lo) * 8) : 0u;
          sg.b = reinterpret_cast<uint64_t>(d.b) + (int64_t(q.fg) * d.n_sensors + s_lo) * d.n_t_pad * int64_t(ROW);
          sg.m = reinterpret_cast<uint64_t>(d.m + (int64_t(q.fg) * d.n_sensors_pad + s_lo) * FB);
          sg.stride = uint64_t(d.n_t_pad) * ROW;
        }
        __syncwarp();
        // Groups of up to S sensors as their windows come, each at most a half or
        // a third of the ring: one long window in a class must not cut every group down to the
        // two sensors that would fit with it.  They end on whole turns of the phases
        // where there are as many.
        uint32_t before = 0;
        for (int i0 = 0; i0 < n && ok;) {
          const int at = i0 + lane;
          const uint32_t u0 = __shfl_sync(0xffffffffu, a0, at & 31), u1 = __shfl_sync(0xffffffffu, a1, at & 31);
          const uint32_t upto = at < 32 ? u0 : u1;  // rows up to this sensor
          const bool in = at < n && int(upto - before) <= cap;
          int se = max(1, __popc(__ballot_sync(0xffffffffu, in)));
          const int turn = i0 & (SW - 1);
          if (turn) se = min(se, SW - turn);
          else if (se > SW) se &= ~(SW - 1);
          const uint32_t to = __shfl_sync(0xffffffffu, upto, se - 1);
          ok = publish(se, i0, sgi, to - before);
          before = to;
          i0 += se;
        }
        if (++sgi == kSegs) sgi = 0;
      }
      t_cur = t_next;
      t_next = __shfl_sync(0xffffffffu, t_next2, 0);
      if (t_next > N) t_next = N;
    }
    // end of work: a slot without data whose unit index is -1, and one for
    // each other copier
    while (ok && n_fly > kSlots - NC) ok = release_oldest();
    if (ok && lane == 0) {
      unit_ring[ju % kRing] = -1;
      for (int c = 0; c < NC; ++c) {
        const int k = (next + c) % kSlots;
        slot_hdr[k] = make_uint4(0u, 0u, 0u, 0u);
        mbar_arrive(&full[k]);
        mbar_arrive(&plan_bar[k]);
      }
    }
    // drain the copies still in flight before the CTA may exit
    for (; n_fly > 0; --n_fly) {
      mbar_wait_bounded(&full[oldest], parity, p.timeout_ns, nullptr);
      if (++oldest == kSlots) {
        oldest = 0;
        parity ^= 1u;
      }
    }
    if (meta_last >= 0)
      mbar_wait_bounded(&meta_bar[meta_last & 1], uint32_t((meta_last >> 1) & 1), p.timeout_ns, nullptr);
  } else {
    // ------------------------------------------------------------ consumers --
    // clear the image outside the mask while the pipeline fills
    for (int i = 0; i < p.n_inst; ++i) {
      const InstDesc& d = p.inst[i];
      const int64_t n = int64_t(d.n_frames) * d.n_zero_runs;
      for (int64_t r = int64_t(blockIdx.x) * NW + warp; r < n; r += int64_t(gridDim.x) * NW) {
        const int f = int(r / d.n_zero_runs), k = int(r - int64_t(f) * d.n_zero_runs);
        const int z0 = __ldcg(d.zero_runs + 2 * k), len = __ldcg(d.zero_runs + 2 * k + 1);
        float* o = d.out + int64_t(f) * d.out_stride + z0;
        for (int i2 = lane; i2 < len; i2 += 32) o[i2] = 0.0f;
      }
    }
    const int lq = lane % LPP, g = lane / LPP;
    // the lane's pixels, V neighbours at a time
    auto pixel = [&](int a) { return warp * NPX + (a / V) * (PPW * V) + g * V + a % V; };
    // Bank conflicts are met within a quarter warp (8 lanes, Q pixels).  With
    // two quads per lane neighbouring pixels take the two halves of their rows
    // in opposite order; FP32 rows that do not fill the banks are taken even
    // or odd one first.
    constexpr int Q = 8 / LPP;
    constexpr bool PAR = FMT == kBF32 && FB < 32;
    constexpr int PB = NQ == 2 ? 2 : (Q > 1 ? Q / 2 : 1);
    const uint32_t odd_first = PAR ? uint32_t(g / PB) & 1u : 0u;
    uint32_t quad[NQ];  // byte offsets of the lane's quads in a row
#pragma unroll
    for (int k = 0; k < NQ; ++k) quad[k] = uint32_t(lq) * 16u + (NQ == 2 ? (uint32_t(k) ^ (uint32_t(g) & 1u)) * (ROW / 2u) : 0u);
    // Computed offsets and weights are the same for the LPP lanes of a pixel: a
    // lane evaluates them for pixels i * 32 + lane of its warp and the lanes of
    // a pixel fetch them by shuffles where that saves evaluations (64 FP32
    // constant-speed frames, 256-pixel tiles: 437 -> 380 us; not for 16-frame
    // rows with computed delays, whose two pixels per lane save too little:
    // 181 us against 191).
    constexpr bool SHARE = A > (NPX + 31) / 32 && (FB != 16 || MODE == 2);
    constexpr int NV = SHARE ? (NPX + 31) / 32 : A;
    auto spread = [&](const float (&mine)[NV], float (&of)[A]) {
#pragma unroll
      for (int a = 0; a < A; ++a) {
        if constexpr (!SHARE) {
          of[a] = mine[a];
          continue;
        }
        const int l = pixel(a) - warp * NPX;
        float v = __shfl_sync(0xffffffffu, mine[0], l & 31);
        if constexpr (SHARE && NV > 1) {
          const float v1 = __shfl_sync(0xffffffffu, mine[1], l & 31);
          v = l < 32 ? v : v1;
        }
        of[a] = v;
      }
    };
    const uint32_t u_lane = uint32_t(warp * NPX + g * V) * 4u;
    int inst = 0;
    int st = 0;             // slot in use and the parity of its next completion
    uint32_t parity = 0;
    bool ok = true;
    auto wait_full = [&]() -> bool {
      if (mbar_wait_bounded(&full[st], parity, p.timeout_ns, abort_flag)) return true;
      if (lane == 0) {
        atomicOr(p.status, kStatusTimeout);
        *abort_flag = 1;
      }
      return false;
    };
    for (int ju = 0; ok; ju = (ju + 1) % kRing) {
      if (!wait_full()) break;
      const int64_t u = unit_ring[ju];
      if (u < 0) break;
      const RowsUnit q = decode_rows(p, u, inst);
      const InstDesc& d = p.inst[q.inst];
      float4 pq[NV];  // constant speed or weights: pixels relative to the tile anchor
      if constexpr (DELAYS != 0 || WGT != 0) {
#pragma unroll
        for (int i = 0; i < NV; ++i) pq[i] = __ldcg(d.pix + int64_t(q.tile) * P + (SHARE ? warp * NPX + (i * 32 + lane) % NPX : pixel(i)));
      }
      bool first = true;
      for (int seg = q.seg0; seg < q.seg1 && ok; ++seg) {
        const int s_lo = seg * d.G, s_hi = min(d.n_sensors, s_lo + d.G);
        f32x2 acc[SW][A][2 * NQ];
#pragma unroll
        for (int ph = 0; ph < SW; ++ph)
#pragma unroll
          for (int a = 0; a < A; ++a)
#pragma unroll
            for (int k = 0; k < 2 * NQ; ++k) acc[ph][a][k] = 0ull;
        for (int s0 = s_lo; s0 < s_hi;) {
          if (!first && !wait_full()) {
            ok = false;
            break;
          }
          first = false;
          const uint4 hdr = slot_hdr[st];
          const int se = int(hdr.y);
          const RowsGroup L(se, P, FB, MODE);
          const uint32_t sb = ring_s + hdr.x;
          const uint32_t m_at = sb + L.m, rec_at = smem_addr(recs + st * kRowsMaxS);
          struct Head {  // what a sensor needs before its rows
            uint2 rec;
            f32x2 m[2 * NQ];
            float uu[A];
          };
          auto load_head = [&](Head& h, int sl) {
            h.rec = lds_u2(rec_at + uint32_t(sl) * 8u);
#pragma unroll
            for (int k = 0; k < NQ; ++k) lds_2x64(m_at + uint32_t(sl) * ROW + quad[k], h.m[2 * k], h.m[2 * k + 1]);
            if constexpr (DELAYS == 0) {
#pragma unroll
              for (int a = 0; a < A; a += V) {
                const uint32_t at = sb + u_lane + uint32_t(sl) * (P * 4u) + uint32_t(a / V) * (PPW * V * 4u);
                if constexpr (V == 4) {
                  const uint4 v = lds_u4(at);
                  h.uu[a] = __uint_as_float(v.x); h.uu[a + 1] = __uint_as_float(v.y);
                  h.uu[a + 2] = __uint_as_float(v.z); h.uu[a + 3] = __uint_as_float(v.w);
                } else if constexpr (V == 2) {
                  const uint2 v = lds_u2(at);
                  h.uu[a] = __uint_as_float(v.x); h.uu[a + 1] = __uint_as_float(v.y);
                } else {
                  h.uu[a] = __uint_as_float(lds_u32(at));
                }
              }
            }
          };
          // sensor sl of the group into the accumulators `ac` of its phase
          auto sensor = [&](f32x2 (&ac)[A][2 * NQ], Head& h, int sl) {
            const uint32_t base = h.rec.x;
            const float lim = __uint_as_float(h.rec.y);
            if constexpr (DELAYS != 0) {
              const float4* sa = reinterpret_cast<const float4*>(ring + hdr.x) + 2 * sl;
              float mine[NV];
              constant_offsets<NV>(mine, pq, sa[0], sa[1]);
              spread(mine, h.uu);
            }
            // floor and phase from the FP32 bits: u + 2^23 rounded toward
            // zero is 2^23 + floor(u), whose low bits are floor(u)
            float ph[A];
            uint32_t row[A], swap[A];
#pragma unroll
            for (int a = 0; a < A; ++a) {
              const float uc = fminf(h.uu[a], lim);
              const float t = __fadd_rz(uc, 8388608.0f);
              ph[a] = __fsub_rn(uc, __fsub_rn(t, 8388608.0f));
              const uint32_t tb = __float_as_uint(t);
              row[a] = base + tb * ROW;
              if constexpr (PAR) {
                // this lane's first row is the even or the odd one of the two
                swap[a] = (tb ^ odd_first) & 1u;
                row[a] += swap[a] * ROW;
              }
            }
            float ww[A];
            if constexpr (WGT != 0) {
              const float4* wa = reinterpret_cast<const float4*>(ring + hdr.x + L.wa) + 2 * sl;
              const float4 E = wa[0], Nn = wa[1];
              float mine[NV];
#pragma unroll
              for (int i = 0; i < NV; ++i) mine[i] = solid_angle_weight(pq[i], E, Nn);
              spread(mine, ww);
            }
#pragma unroll
            for (int a = 0; a < A; ++a) {
              f32x2 wp = 0ull;
              if constexpr (WGT != 0) wp = pack2(ww[a], ww[a]);
              // swapped rows: x is b_{k+1} and y is b_k, so y - x is the exact
              // negative of the slope and the phase changes sign with it
              const float sp = PAR ? __uint_as_float(__float_as_uint(ph[a]) ^ (swap[a] << 31)) : ph[a];
              const f32x2 php = pack2(sp, sp);
#pragma unroll
              for (int k = 0; k < NQ; ++k) {
                const uint32_t r = row[a] + quad[k];
                f32x2 v0, v1;
                if constexpr (FMT == kBF32) {
                  f32x2 x0, x1, y0, y1;
                  lds_2x64(r, x0, x1);
                  if constexpr (PAR) {
                    lds_2x64(r + ROW - swap[a] * (2u * ROW), y0, y1);
                    v0 = fma2(php, sub2(y0, x0), swap[a] ? y0 : x0);
                    v1 = fma2(php, sub2(y1, x1), swap[a] ? y1 : x1);
                  } else {
                    lds_2x64(r + ROW, y0, y1);
                    v0 = fma2(php, sub2(y0, x0), x0);
                    v1 = fma2(php, sub2(y1, x1), x1);
                  }
                } else {
                  const uint4 w = lds_u4(r);
                  if constexpr (FMT == kBBF16P) {
                    v0 = fma2(php, pack2u(w.x & 0xffff0000u, w.y & 0xffff0000u), pack2u(w.x << 16, w.y << 16));
                    v1 = fma2(php, pack2u(w.z & 0xffff0000u, w.w & 0xffff0000u), pack2u(w.z << 16, w.w << 16));
                  } else {
                    const float2 h0 = __half22float2(*reinterpret_cast<const __half2*>(&w.x));
                    const float2 h1 = __half22float2(*reinterpret_cast<const __half2*>(&w.y));
                    const float2 h2 = __half22float2(*reinterpret_cast<const __half2*>(&w.z));
                    const float2 h3 = __half22float2(*reinterpret_cast<const __half2*>(&w.w));
                    v0 = fma2(php, pack2(h0.y, h1.y), pack2(h0.x, h1.x));
                    v1 = fma2(php, pack2(h2.y, h3.y), pack2(h2.x, h3.x));
                  }
                }
                if constexpr (WGT != 0) {
                  v0 = mul2(wp, v0);
                  v1 = mul2(wp, v1);
                }
                ac[a][2 * k] = fma2(h.m[2 * k], v0, ac[a][2 * k]);
                ac[a][2 * k + 1] = fma2(h.m[2 * k + 1], v1, ac[a][2 * k + 1]);
              }
            }
          };
          // sensor sl of the group has phase (s0 - s_lo + sl) mod SW; groups are
          // whole turns of the phases but where windows are long
          const int ph0 = (s0 - s_lo) & (SW - 1);
          s0 += se;
          if (ph0 == 0 && (se & (SW - 1)) == 0) {
            for (int k = 0; k < se; k += SW) {
#pragma unroll
              for (int ph = 0; ph < SW; ph += 2) {
                Head h0, h1;
                load_head(h0, k + ph);
                load_head(h1, k + ph + 1);
                sensor(acc[ph], h0, k + ph);
                sensor(acc[ph + 1], h1, k + ph + 1);
              }
            }
          } else {
            for (int k = -ph0; k < se; k += SW) {
#pragma unroll
              for (int ph = 0; ph < SW; ++ph) {
                if (unsigned(k + ph) >= unsigned(se)) continue;
                Head h;
                load_head(h, k + ph);
                sensor(acc[ph], h, k + ph);
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[st]);
          if (++st == kSlots) {
            st = 0;
            parity ^= 1u;
          }
        }
        if (!ok) break;
        // the segment's sums: phases in order; then the segments in order
#pragma unroll
        for (int a = 0; a < A; ++a) {
          const int px = pixel(a);
#pragma unroll
          for (int k = 0; k < NQ; ++k) {
            const int fq = int(quad[k] / 4u);  // first of the quad's frames
            float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int ph = 0; ph < SW; ++ph) {
              float x[4];
              unpack2(acc[ph][a][2 * k], x[0], x[1]);
              unpack2(acc[ph][a][2 * k + 1], x[2], x[3]);
#pragma unroll
              for (int i = 0; i < 4; ++i) v[i] += x[i];
            }
            if (p.split && d.n_seg > 1) {
              float* part = d.part + (((int64_t(q.fg) * d.n_tiles + q.tile) * d.n_seg + seg) * P + px) * FB + fq;
              __stcg(reinterpret_cast<float4*>(part), make_float4(v[0], v[1], v[2], v[3]));
              continue;
            }
            if (d.n_seg > 1) {
              float4* tp = reinterpret_cast<float4*>(total + px * FB + fq);  // this lane's own
              float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
              if (seg > 0) t = *tp;
              t.x += v[0]; t.y += v[1]; t.z += v[2]; t.w += v[3];
              if (seg + 1 < d.n_seg) {
                *tp = t;
                continue;
              }
              v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
            }
            const int o = __ldcg(d.slot + int64_t(q.tile) * P + px);
            const int f0 = q.fg * FB + fq;
            if (o >= 0) {
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (f0 + i < d.n_frames) d.out[int64_t(f0 + i) * d.out_stride + o] = v[i];
            }
          }
        }
      }
    }
  }
  // the last CTA out resets the unit tickets for the next launch
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(p.sched + 2, 1u) == gridDim.x - 1) {
      atomicExch(reinterpret_cast<unsigned long long*>(p.sched), 0ull);
      atomicExch(p.sched + 2, 0u);
    }
  }
}

// Sum of the segment sums of a split launch, in segment order, written to the
// image.  FB / 4 neighbouring lanes take the frames of one pixel (16 bytes
// each): whole rows of the partial sums are read; 8 segments are in flight.
// Lanes of rows of 16 and 32 frames hold few neighbouring pixels of a frame; their
// sums are turned in shared memory, so that a warp writes 32 (into an image in host
// memory, pieces of 4 pixels took 122 us for 32 frames of 21 300; small launches
// with short rows would only lose a microsecond).
template <int FB>
__global__ void __launch_bounds__(256) rows_reduce_kernel(const __grid_constant__ StreamParams p, int P) {
  constexpr int LPP = FB / 4, K = 8;
  constexpr bool TURN = FB >= 16;
  constexpr int PX = 256 / LPP, PITCH = PX + 8 / LPP;  // pixels of one pass; no bank twice
  __shared__ float turned[TURN ? FB : 1][TURN ? PITCH : 1];
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int i = 0; i < p.n_inst; ++i) {
    const InstDesc& d = p.inst[i];
    if (d.n_seg == 1) continue;  // written by the gather
    const int64_t n = int64_t(d.n_fg) * d.n_tiles * P;  // pixels of all frame groups
    for (int64_t first = int64_t(blockIdx.x) * PX; first < n; first += int64_t(gridDim.x) * PX) {
      // what this thread adds: a quad of frames of a pixel; what it writes: that,
      // or the frames f0, f0 + LPP, .. of another
      const int lq = int(threadIdx.x) % LPP, mine = int(threadIdx.x) / LPP;
      const int at = TURN ? int(threadIdx.x) % PX : mine, f0 = TURN ? int(threadIdx.x) / PX : lq * 4;
      int o = -1, fg = 0;
      if (first + at < n) {
        fg = int((first + at) / P / d.n_tiles);
        o = __ldcg(d.slot + first + at - int64_t(fg) * d.n_tiles * P);
      }
      float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (first + mine < n) {
        const int64_t ft = (first + mine) / P;  // frame group * n_tiles + tile
        const int px = int(first + mine - ft * P);
        const float4* src = reinterpret_cast<const float4*>(d.part + (ft * d.n_seg * P + px) * FB) + lq;
        const int64_t step = int64_t(P) * LPP;
        for (int s0 = 0; s0 < d.n_seg; s0 += K) {
          float4 x[K];
#pragma unroll
          for (int k = 0; k < K; ++k)
            x[k] = s0 + k < d.n_seg ? __ldcg(src + (s0 + k) * step) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int k = 0; k < K; ++k) {
            if (s0 + k >= d.n_seg) break;
            t.x += x[k].x; t.y += x[k].y; t.z += x[k].z; t.w += x[k].w;
          }
        }
      }
      float v[4] = {t.x, t.y, t.z, t.w};
      if constexpr (TURN) {
#pragma unroll
        for (int k = 0; k < 4; ++k) turned[lq * 4 + k][mine] = v[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = turned[f0 + k * LPP][at];
        __syncthreads();
      }
      if (o < 0) continue;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int f = fg * FB + f0 + (TURN ? k * LPP : k);
        if (f < d.n_frames) d.out[int64_t(f) * d.out_stride + o] = v[k];
      }
    }
  }
}

// ------------------------------------------------------- launch templates --
template <int P, int FB, int FMT, int SW, int MODE>
static cudaError_t rows_t(const StreamParams& p, size_t smem, int grid, cudaStream_t st, int* resident,
                          int n_sm) {
  using SH = RowsShape<P, FB, FMT, MODE>;
  auto kern = gather_rows_kernel<P, FB, FMT, SW, MODE>;
  static SmemGrant grant;
  if (cudaError_t e = grant_smem(grant, kern, smem); e != cudaSuccess) return e;
  if (resident) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, SH::THREADS, smem);
    if (e != cudaSuccess) return e;
    *resident = per_sm * n_sm;
    return cudaSuccess;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(SH::THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

// Launch (grid > 0), count resident CTAs (resident != nullptr) or name the
// kernel (func != nullptr) of the instantiation that matches the config.
template <int P, int FB, int FMT, int SW, int MODE>
static cudaError_t rows_do(const StreamParams* p, size_t smem, int grid, cudaStream_t st, int* resident,
                           int n_sm, const void** func) {
  if (func) {
    *func = reinterpret_cast<const void*>(gather_rows_kernel<P, FB, FMT, SW, MODE>);
    return cudaSuccess;
  }
  return rows_t<P, FB, FMT, SW, MODE>(*p, smem, grid, st, resident, n_sm);
}

template <int P, int FMT, int SW, int MODE>
static cudaError_t rows_fb(int FB, const StreamParams* p, size_t smem, int grid, cudaStream_t st,
                           int* resident, int n_sm, const void** func) {
  switch (FB) {
    case 4: return rows_do<P, 4, FMT, SW, MODE>(p, smem, grid, st, resident, n_sm, func);
    case 8: return rows_do<P, 8, FMT, SW, MODE>(p, smem, grid, st, resident, n_sm, func);
    case 16: return rows_do<P, 16, FMT, SW, MODE>(p, smem, grid, st, resident, n_sm, func);
    case 32: return rows_do<P, 32, FMT, SW, MODE>(p, smem, grid, st, resident, n_sm, func);
    default: return cudaErrorInvalidValue;
  }
}

template <int MODE>
static cudaError_t rows_dispatch_t(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem,
                                   int grid, cudaStream_t st, int* resident, const void** func) {
  const int n_sm = c.n_sm;
  if (c.P == 128 && c.SW == 4) {
    if (fmt == kBF32) return rows_fb<128, kBF32, 4, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
    if (fmt == kBBF16P) return rows_fb<128, kBBF16P, 4, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
    if (fmt == kBF16P) return rows_fb<128, kBF16P, 4, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
  } else if (c.P == 256 && c.SW == 2) {
    if (fmt == kBF32) return rows_fb<256, kBF32, 2, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
    if (fmt == kBBF16P) return rows_fb<256, kBBF16P, 2, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
    if (fmt == kBF16P) return rows_fb<256, kBF16P, 2, MODE>(c.FB, p, smem, grid, st, resident, n_sm, func);
  }
  return cudaErrorInvalidValue;
}

// One translation unit per mode, so the families compile in parallel.
cudaError_t rows_dispatch_0(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func);
cudaError_t rows_dispatch_1(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func);
cudaError_t rows_dispatch_2(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func);
cudaError_t rows_dispatch_3(const GatherConfig& c, int fmt, const StreamParams* p, size_t smem, int grid,
                            cudaStream_t st, int* resident, const void** func);

}  // namespace patbp
