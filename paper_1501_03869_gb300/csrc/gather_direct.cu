// gather_direct.cu -- the single-frame gather of Eq. (BP) without the staged
// pipeline.
//
// Two gathers share the reduction kernel below.  gather_window_kernel (windows
// that fit a slot, and launches that fill its CTAs: window_pays in row_rules.h)
// copies each sensor's integrand window into shared memory per warp and
// interpolates there; gather_direct_kernel, described next, gathers from L2 and
// takes every other case.  Both give the same bits.
//
// Two launches.  The gather kernel is persistent: CTA c takes units (tile,
// segment of G sensors) c, c + grid, c + 2 grid, ... in tile-major order, and
// (constant speed) asks L2 for each unit's delay data two units ahead with one
// bulk prefetch.
// Its warps are the (pixel group, sensor phase) pairs of the staged kernel's
// consumers; a warp reads the delay data (table offsets, or the constant-
// speed anchors) and the window bases for a chunk of its sensors, then
// gathers the integrand rows from L2 with loads that never branch (an arrival
// after the record reads a zero padding row), and finally stores its phase
// sums -- no barrier, fence or atomic anywhere, so no warp ever waits for
// another.  The reduction kernel then forms every pixel's sum over phases and
// segments and scatters it to the image.
//
// Both kernels are launched as programmatic dependents, which can start before
// the kernels ahead of them in the stream have finished; lines that an earlier
// kernel left in an SM's L1 are then not reliably dropped, so every global load
// here goes through L2 only (ld.global.cg), never the non-coherent L1 path.
//
// Arithmetic and summation order are those of the staged kernel with one
// frame per unit (gather.cuh): phase sp of a segment accumulates sensors
// s_lo + sp, s_lo + sp + SW, ... with acc = fma(m_s, fma(ph, b1 - b0, b0), acc),
// phases are summed in order 0..SW-1 and segments in order 0..n_seg-1.  A frame
// therefore gives the same bits here as inside any batch that the staged kernel
// reconstructs.
//
// With solid-angle weights (WGT = 1, the exact back projection of Sec. II-C)
// each term carries its own weight w(pixel, sensor), evaluated from the
// sensor's 32-byte weight anchor and the pixel's position terms by the same
// function as the staged kernel: acc = fma(m_s, w * lerp, acc).
#include <algorithm>

#include "gather.cuh"
#include "packed.cuh"
#include "row_rules.h"

namespace patbp {

namespace {

constexpr int kDirectChunk = 1;    // sensors of a phase whose loads are issued together
constexpr int kDirectMinCtas = 8;  // resident CTAs per SM the registers must allow

struct DirectParams {
  const float* u;
  const float* anchor;
  const float4* pix;
  const float* wanchor;
  const int32_t* base;
  const int32_t* slot;
  const int32_t* zero_runs;
  const void* b;
  const float* m;
  float* out;
  float* part;  // [n_tiles][n_seg][SW][P] phase sums
  int* status;
  int* host_status;  // the reduction copies *status here when set
  uint64_t timeout_ns;  // bound of every device-side wait
  int n_zero_runs, n_sensors, n_sensors_pad, n_t_pad, n_tiles, n_seg, G;
  int W;  // longest window of one (tile, sensor) (rows)
};

// One sensor's contribution to this lane's 4 pixels; `row` points at the
// sensor's window base in the integrand.  Offsets above `cap` are after the
// record: they read the zero row `zrow` (a padding row after the record) with
// phase 0, which adds m * 0 exactly as the staged kernel's zero rows do.
template <int FMT, int WGT>
__device__ __forceinline__ void direct_accumulate(float (&acc)[4], const float (&uu)[4], float cap,
                                                  const uint32_t* row, unsigned zrow, float mm,
                                                  const float (&ww)[4]) {
#pragma unroll
  for (int x = 0; x < 4; ++x) {
    const bool in = uu[x] <= cap;
    const unsigned t = unsigned(__float2int_rz(uu[x]));
    const unsigned i = in ? t : zrow;
    const float ph = in ? uu[x] - float(t) : 0.0f;
    const uint32_t w0 = __ldcg(row + i);
    float v;
    if constexpr (FMT == kBF32) {
      const float b0 = __uint_as_float(w0), b1 = __uint_as_float(__ldcg(row + i + 1));
      v = fmaf(ph, b1 - b0, b0);
    } else if constexpr (FMT == kBBF16P) {
      v = fmaf(ph, __uint_as_float(w0 & 0xffff0000u), __uint_as_float(w0 << 16));
    } else {
      const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&w0));
      v = fmaf(ph, h.y, h.x);
    }
    if constexpr (WGT != 0) v = __fmul_rn(ww[x], v);
    acc[x] = fmaf(mm, v, acc[x]);
  }
}

__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Pull the delay data of `unit` (one contiguous block) into L2.
template <int P, int DELAYS>
__device__ __forceinline__ void prefetch_unit(const DirectParams& p, int64_t unit, int64_t n_units) {
  if (unit >= n_units) return;
  const int tile = int(unit / p.n_seg), seg = int(unit - int64_t(tile) * p.n_seg);
  const int s_lo = seg * p.G, n = min(p.n_sensors, s_lo + p.G) - s_lo;
  if constexpr (DELAYS == 0)
    bulk_prefetch_l2(p.u + (int64_t(tile) * p.n_sensors + s_lo) * P, uint32_t(n) * P * 4);
  else
    bulk_prefetch_l2(p.anchor + (int64_t(tile) * p.n_sensors_pad + s_lo) * 8, uint32_t(n) * 32);
}

template <int P, int SW, int FMT, int DELAYS, int WGT>
__global__ void __launch_bounds__(32 * (P / 128) * SW, kDirectMinCtas)
    gather_direct_kernel(const __grid_constant__ DirectParams p) {
  constexpr int PW = P / 128;
  constexpr int CH = kDirectChunk;
  // the reduction kernel may start now; it waits for this grid's results
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pg = warp % PW, sp = warp / PW;
  const int px0 = pg * 128 + lane;
  const int64_t n_units = int64_t(p.n_tiles) * p.n_seg;
  if (DELAYS != 0 && threadIdx.x == 0) {
    prefetch_unit<P, DELAYS>(p, blockIdx.x, n_units);
    prefetch_unit<P, DELAYS>(p, int64_t(blockIdx.x) + gridDim.x, n_units);
  }
  const uint32_t* bsrc = static_cast<const uint32_t*>(p.b);
  bool waited = false;
  for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
    if (DELAYS != 0 && threadIdx.x == 0)
      prefetch_unit<P, DELAYS>(p, unit + 2 * int64_t(gridDim.x), n_units);
    const int tile = int(unit / p.n_seg);
    const int seg = int(unit - int64_t(tile) * p.n_seg);
    const int s_lo = seg * p.G, s_hi = min(p.n_sensors, s_lo + p.G);
    float4 pq[4];
    if constexpr (DELAYS != 0 || WGT != 0) {
#pragma unroll
      for (int x = 0; x < 4; ++x) pq[x] = __ldcg(p.pix + int64_t(tile) * P + px0 + x * 32);
    }
    const float4* wrow = WGT != 0 ? reinterpret_cast<const float4*>(p.wanchor) +
                                        int64_t(tile) * p.n_sensors_pad * 2
                                  : nullptr;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float ww[4] = {1.0f, 1.0f, 1.0f, 1.0f};
    if constexpr (DELAYS == 0) {
      // Table offsets: one sensor at a time, software-pipelined -- the next
      // sensor's offsets and window base are in flight while this one
      // gathers (the first ones before waiting for the preprocessing grid).
      float un[4];
      uint32_t bn = 0u;
      float4 wn0 = make_float4(0.f, 0.f, 0.f, 0.f), wn1 = wn0;
      auto load_next = [&](int s) {
        bn = uint32_t(__ldcg(p.base + int64_t(tile) * p.n_sensors_pad + s));
        const float* urow = p.u + (int64_t(tile) * p.n_sensors + s) * P + px0;
#pragma unroll
        for (int x = 0; x < 4; ++x) un[x] = __ldcg(urow + x * 32);
        if constexpr (WGT != 0) {
          wn0 = __ldcg(wrow + 2 * s);
          wn1 = __ldcg(wrow + 2 * s + 1);
        }
      };
      if (s_lo + sp < s_hi) load_next(s_lo + sp);
      for (int s = s_lo + sp; s < s_hi; s += SW) {
        const float uu[4] = {un[0], un[1], un[2], un[3]};
        const unsigned bs = bn & 0xffffu;
        if constexpr (WGT != 0) solid_angle_weights(ww, pq, wn0, wn1);
        if (s + SW < s_hi) load_next(s + SW);
        if (!waited) {
          // integrand and multipliers come from the preprocessing grid
          asm volatile("griddepcontrol.wait;" ::: "memory");
          waited = true;
        }
        const float mm = __ldcg(p.m + s);
        const uint32_t* row = bsrc + int64_t(s) * p.n_t_pad + bs;
        direct_accumulate<FMT, WGT>(acc, uu, 1.0e29f, row, unsigned(p.n_t_pad - 1) - bs, mm, ww);
      }
    } else {
      // Sensors of this phase in chunks of CH: the loads that do not depend on
      // the preprocessing (delay data, window bases) are issued for the chunk
      // first -- for the first chunk before waiting for the preprocessing grid.
      for (int c0 = s_lo + sp; c0 < s_hi; c0 += CH * SW) {
        uint32_t bw[CH];
        float uu[CH][4];
        float4 an[CH][2];
        float4 wa[WGT ? CH : 1][2];
  #pragma unroll
        for (int j = 0; j < CH; ++j) {
          const int s = c0 + j * SW;
          const bool ok = s < s_hi;
          bw[j] = ok ? uint32_t(__ldcg(p.base + int64_t(tile) * p.n_sensors_pad + s)) : 0u;
          const float4* ap = reinterpret_cast<const float4*>(p.anchor) +
                             (int64_t(tile) * p.n_sensors_pad + (ok ? s : s_lo)) * 2;
          an[j][0] = __ldcg(ap);
          an[j][1] = __ldcg(ap + 1);
          if (!ok) an[j][1].y = -1.0f;  // cap below every offset: nothing to add
          if constexpr (WGT != 0) {
            wa[j][0] = __ldcg(wrow + 2 * (ok ? s : s_lo));
            wa[j][1] = __ldcg(wrow + 2 * (ok ? s : s_lo) + 1);
          }
        }
        if (!waited) {
          // integrand and multipliers come from the preprocessing grid
          asm volatile("griddepcontrol.wait;" ::: "memory");
          waited = true;
        }
        float mm[CH];
  #pragma unroll
        for (int j = 0; j < CH; ++j) mm[j] = c0 + j * SW < s_hi ? __ldcg(p.m + c0 + j * SW) : 0.0f;
  #pragma unroll
        for (int j = 0; j < CH; ++j) {
          const int s = min(c0 + j * SW, s_hi - 1);
          const float4 A = an[j][0], B = an[j][1];
          if (B.w == 0.0f) {
            const float m2u0 = -2.0f * A.w;
  #pragma unroll
            for (int x = 0; x < 4; ++x) {
              const float num =
                  fmaf(pq[x].x, A.x, fmaf(pq[x].y, A.y, fmaf(pq[x].z, A.z, pq[x].w)));
              const float sq = num + B.z;
              const float y = rsqrtf(sq);
              const float da = sq * y - A.w;
              const float r = fmaf(-da, da, fmaf(m2u0, da, num));
              const float v = fmaf(r, 0.5f * y, da) + B.x;
              uu[j][x] = v > B.y ? kFarOffset : fmaxf(v, 0.0f);
            }
          } else {
  #pragma unroll
            for (int x = 0; x < 4; ++x) {
              const float d0 = fmaf(0.5f, pq[x].x, A.x), d1 = fmaf(0.5f, pq[x].y, A.y),
                          d2 = fmaf(0.5f, pq[x].z, A.z);
              const float sq = fmaxf(fmaf(d0, d0, fmaf(d1, d1, d2 * d2)), 1.0e-30f);
              const float v = (sq * rsqrtf(sq) - A.w) + B.x;
              uu[j][x] = v > B.y ? kFarOffset : fmaxf(v, 0.0f);
            }
          }
          const unsigned bs = bw[j] & 0xffffu;
          const uint32_t* row = bsrc + int64_t(s) * p.n_t_pad + bs;
          if constexpr (WGT != 0) solid_angle_weights(ww, pq, wa[j][0], wa[j][1]);
          direct_accumulate<FMT, WGT>(acc, uu[j], 1.0e29f, row, unsigned(p.n_t_pad - 1) - bs, mm[j],
                                      ww);
        }
      }
    }
    float* dst = p.part + ((int64_t(tile) * p.n_seg + seg) * SW + sp) * P + px0;
#pragma unroll
    for (int x = 0; x < 4; ++x) dst[x * 32] = acc[x];
  }
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Clears the image outside the mask.  The warps of the grid share the runs (of
// at most 512 nodes), up to 32 at a time: a lane loads each run's ends, so a warp
// waits for memory once and not once per run.  Frame of 64 sensors, 2 000 of 256 x
// 256 nodes imaged (16 CTAs): 9.4 us with a CTA per run of any length, 8.5 with
// lanes loading the ends, 6.8 with short runs too.
__device__ __forceinline__ void clear_outside(const DirectParams& p) {
  const int warps = int(gridDim.x * blockDim.x) >> 5, lane = threadIdx.x & 31;
  const int warp = int(blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int per = min(32, (p.n_zero_runs + warps - 1) / warps);
  for (int64_t r0 = int64_t(warp) * per; r0 < p.n_zero_runs; r0 += int64_t(warps) * per) {
    const int n = int(min(int64_t(per), p.n_zero_runs - r0));
    int st0 = 0, len = 0;
    if (lane < n) {
      st0 = p.zero_runs[2 * (r0 + lane)];
      len = p.zero_runs[2 * (r0 + lane) + 1];
    }
    for (int k = 0; k < n; ++k) {
      const int at = __shfl_sync(0xffffffffu, st0, k), e = __shfl_sync(0xffffffffu, len, k);
      for (int i = lane; i < e; i += 32) p.out[at + i] = 0.0f;
    }
  }
}

// Sum of every pixel over phases (in order) and segments (in order), written
// to its place in the image (SW = 1: the part buffer holds segment sums); also clears the image outside the mask.  The
// loads of 8 segments are issued before their sums, so a pixel costs about
// one L2 round trip per 8 segments.
template <int P, int SW>
__global__ void __launch_bounds__(256) direct_reduce_kernel(const __grid_constant__ DirectParams p) {
  constexpr int K = 8;
  clear_outside(p);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // the kernels before this one are complete: their status is final
  if (p.host_status && blockIdx.x == 0 && threadIdx.x == 0) *p.host_status = __ldcg(p.status);
  const int64_t n = int64_t(p.n_tiles) * P;
  for (int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; idx < n;
       idx += int64_t(gridDim.x) * blockDim.x) {
    const int o = __ldcg(p.slot + idx);
    const int64_t tile = idx / P;
    const int q = int(idx - tile * P);
    const float* src = p.part + tile * p.n_seg * SW * P + q;
    float t = 0.0f;
    for (int s0 = 0; s0 < p.n_seg; s0 += K) {
      // (the first batch is loaded together with the slot, before its test)
      float x[K][SW];
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int ph = 0; ph < SW; ++ph)
          x[k][ph] = s0 + k < p.n_seg ? __ldcg(src + (int64_t(s0 + k) * SW + ph) * P) : 0.0f;
      if (o < 0) break;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (s0 + k >= p.n_seg) break;
        if constexpr (SW == 1) {
          t += x[k][0];  // phases already summed, in the same order, by the gather
        } else {
          float v = 0.0f;
#pragma unroll
          for (int ph = 0; ph < SW; ++ph) v += x[k][ph];
          t += v;
        }
      }
    }
    if (o >= 0) p.out[o] = t;
  }
}

// ------------------------------------------------------ windowed variant --
// For handles whose every window fits a shared-memory slot of WB rows.  The
// four warps of a CTA are the four (pixel group, sensor phase) pairs of one
// unit, as above; a lane owns 4 neighbouring pixels of its warp's 128
// (their offsets are one 16-byte load; pixels 32 apart met fewer bank conflicts,
// 1.6 to 2.0 wavefronts per load against 2.2 to 2.5, but took 252 us instead of
// 229 on a BF16 volume).  A warp
// takes its sensors two at a time.  For each sensor it copies the tile's
// integrand window (rows base .. base + len) into a slot of its own with
// 16-byte cp.async copies, two steps ahead, while its lanes' table offsets come
// from global memory one step ahead; constant-
// speed delays and solid-angle weights are evaluated from anchors staged in
// shared memory once per unit.  The interpolation then reads shared memory.
// Each slot ends in 8 zero rows at row WB: an offset after the record (the
// table's out-of-record value) is clamped to WB, which gives phase 0 and the
// zero rows, so it adds m * 0 as in the kernel above; so does the absent
// second sensor of a last step.  The CTA sums its four phase sums per pixel in
// order before storing, so the reduction kernel sums segments only; with one
// segment per tile (at most 64 sensors) the sums go to the image and there is no
// reduction launch.
// Arithmetic and summation order are those of gather_direct_kernel: the image
// has the same bits.
//
// What bounds it: instruction issue and shared-memory wavefronts (one warp-sensor
// took 113 instructions at 76 % issue-active with scalar FP32), so
// pixels go through packed FP32 pairs, steps alternate between two register
// sets and two slots with constant addresses, and nothing branches per sensor:
// 84 instructions.  One frame of 512 sensors x 0.6 M voxels (1.24 GB table):
// FP32 301 -> 286 us, BF16 296 -> 243, constant speed 549 -> 422.
//
// Offsets in the window are found from the FP32 bits: for 0 <= u < 2^23,
// u + 2^23 rounded toward zero is 2^23 + floor(u) exactly, its bit pattern is
// 0x4B000000 + floor(u), and (u + 2^23) - 2^23 = floor(u) exactly.
constexpr int kWindowMaxRows = 384;  // largest slot (rows); longer windows take the kernel above

template <int P, int SW, int FMT, int WB, int DELAYS, int WGT>
__global__ void __launch_bounds__(128, window_ctas(DELAYS, WGT, WB))
    gather_window_kernel(const __grid_constant__ DirectParams p) {
  constexpr int PW = P / 128;
  static_assert(PW * SW == 4, "a unit is four warps");
  constexpr int SLOT = WB + 8;  // rows of one slot: window, then 8 zero rows
  constexpr int NC = (WB + 127) / 128;  // 16-byte copies per lane for one window
  constexpr int MAXJ = 64 / SW;         // sensors of a warp (segments of at most 64)
  __shared__ __align__(16) uint32_t swin[4][4][SLOT];
  __shared__ __align__(16) uint2 sbm[4][MAXJ];  // (window base word, multiplier) per sensor of the warp
  __shared__ __align__(16) float4 sanchor[DELAYS ? 4 : 1][DELAYS ? MAXJ : 1][2];
  __shared__ __align__(16) float4 swanchor[WGT ? 4 : 1][WGT ? MAXJ : 1][2];
  __shared__ __align__(16) float ssum[SW][P];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pg = warp % PW, sp = warp / PW;
  const int px0 = pg * 128 + 4 * lane;
  uint32_t* ring = &swin[warp][0][0];
  ring[(lane >> 3) * SLOT + WB + (lane & 7)] = 0u;  // 4 slots x 8 zero rows
  const uint32_t ring_s = smem_addr(ring);
  const int64_t n_units = int64_t(p.n_tiles) * p.n_seg;
  const uint32_t* bsrc = static_cast<const uint32_t*>(p.b);
  const uint32_t bm_s = smem_addr(sbm[warp]);
  const f32x2 magic = pack2(8388608.0f, 8388608.0f), unmagic = pack2(-8388608.0f, -8388608.0f);
  // one segment per tile: its sums are the image, and no reduction follows
  const bool final = p.out && p.n_seg == 1;
  if (final) clear_outside(p);
  // integrand and multipliers come from the preprocessing grid
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (final && p.host_status && blockIdx.x == 0 && threadIdx.x == 0) *p.host_status = __ldcg(p.status);
  for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
    const int tile = int(unit / p.n_seg);
    const int seg = int(unit - int64_t(tile) * p.n_seg);
    const int s_lo = seg * p.G, s_hi = min(p.n_sensors, s_lo + p.G);
    const int s0 = s_lo + sp;  // this warp's sensors: s0, s0 + SW, ...
    const int nj = s0 < s_hi ? (s_hi - s0 + SW - 1) / SW : 0;
    const float* ubase = nullptr;
    if constexpr (DELAYS == 0) {
      ubase = p.u + (int64_t(tile) * p.n_sensors + s0) * P + px0;
      if (unit != int64_t(blockIdx.x) && threadIdx.x == 0) {
        // a CTA's later units (launches with more units than resident CTAs)
        // start at staggered times: their table block is asked into L2 at once.
        // (Not the first unit: every CTA asking for its block at the launch's
        // start delayed the first offsets behind the whole table.)
        bulk_prefetch_l2(p.u + (int64_t(tile) * p.n_sensors + s_lo) * P, uint32_t(s_hi - s_lo) * P * 4);
      }
    }
    const uint32_t* wsrc = bsrc + int64_t(s0) * p.n_t_pad + lane * 4;
    const uint32_t wstep = uint32_t(SW) * uint32_t(p.n_t_pad);
    float4 pq[4];
    if constexpr (DELAYS != 0 || WGT != 0) {
#pragma unroll
      for (int x = 0; x < 4; ++x) pq[x] = __ldcg(p.pix + int64_t(tile) * P + px0 + x);
    }
    // the lane's offsets of the sensors j, j + 1 (past the last: after the record)
    auto load_u = [&](int j, float4 (&d)[2]) {
      if constexpr (DELAYS == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          d[h] = j + h < nj ? __ldcg(reinterpret_cast<const float4*>(ubase + (j + h) * (SW * P)))
                            : make_float4(kFarOffset, kFarOffset, kFarOffset, kFarOffset);
      }
    };
    float4 ua[2], ub[2];
    load_u(0, ua);  // in flight with the window bases below
    if (lane < MAXJ) {
      const int s = s0 + lane * SW;
      uint2 w = make_uint2(0u, 0u);
      if (lane < nj)
        w = make_uint2(uint32_t(__ldcg(p.base + int64_t(tile) * p.n_sensors_pad + s)),
                       __float_as_uint(__ldcg(p.m + s)));
      sbm[warp][lane] = w;
      if constexpr (DELAYS != 0) {
        const float4* ap = reinterpret_cast<const float4*>(p.anchor) +
                           (int64_t(tile) * p.n_sensors_pad + min(s, s_hi - 1)) * 2;
        float4 A = __ldcg(ap), B = __ldcg(ap + 1);
        if (lane >= nj) B.y = -1.0f;  // cap below every offset: nothing to add
        sanchor[warp][lane][0] = A;
        sanchor[warp][lane][1] = B;
      }
      if constexpr (WGT != 0) {
        const float4* wp = reinterpret_cast<const float4*>(p.wanchor) +
                           (int64_t(tile) * p.n_sensors_pad + min(s, s_hi - 1)) * 2;
        swanchor[warp][lane][0] = __ldcg(wp);
        swanchor[warp][lane][1] = __ldcg(wp + 1);
      }
    }
    __syncwarp();
    // windows of the sensors j, j + 1 into the slots 2 buf, 2 buf + 1; one group per step
    auto issue = [&](int j, int buf) {
      if (j < nj) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t b = lds_u32(bm_s + uint32_t(j + h) * 8u);
          const int len = int(b >> 16);
          const uint32_t* src = wsrc + (uint32_t(j + h) * wstep + (b & 0xffffu));
          const uint32_t sa = ring_s + uint32_t(((2 * buf + h) * SLOT + lane * 4) * 4);
#pragma unroll
          for (int c = 0; c < NC; ++c)
            if (lane * 4 + c * 128 < len) cp_async16(sa + c * 512, src + c * 128);
        }
      }
      cp_async_commit();
    };
    issue(0, 0);
    issue(2, 1);
    f32x2 acc[2] = {0ull, 0ull};
    // sensor j, offsets u, slot; the slot's row 0 minus 4 * 0x4B000000 (shared
    // addresses wrap modulo 2^32)
    auto sensor = [&](int j, float4 u4, int slot, float m) {
      float uu[4] = {u4.x, u4.y, u4.z, u4.w};
      if constexpr (DELAYS != 0) constant_offsets<4>(uu, pq, sanchor[warp][j][0], sanchor[warp][j][1]);
      float ww[4];
      if constexpr (WGT != 0) solid_angle_weights(ww, pq, swanchor[warp][j][0], swanchor[warp][j][1]);
      const uint32_t wadj = ring_s + uint32_t(slot * SLOT * 4) - 4u * 0x4B000000u;
      const f32x2 mm = pack2(m, m);
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const f32x2 uc = pack2(fminf(uu[2 * x], float(WB)), fminf(uu[2 * x + 1], float(WB)));
        const f32x2 t = add2_rz(uc, magic);
        const f32x2 ph = sub2(uc, add2(t, unmagic));
        float t0, t1;
        unpack2(t, t0, t1);
        const uint32_t a0 = wadj + 4u * __float_as_uint(t0), a1 = wadj + 4u * __float_as_uint(t1);
        f32x2 v;
        if constexpr (FMT == kBF32) {
          const f32x2 b0 = pack2u(lds_u32(a0), lds_u32(a1)), b1 = pack2u(lds_u32(a0 + 4), lds_u32(a1 + 4));
          v = fma2(ph, sub2(b1, b0), b0);
        } else {
          const uint32_t w0 = lds_u32(a0), w1 = lds_u32(a1);
          if constexpr (FMT == kBBF16P) {
            v = fma2(ph, pack2u(w0 & 0xffff0000u, w1 & 0xffff0000u), pack2u(w0 << 16, w1 << 16));
          } else {
            const float2 h0 = __half22float2(*reinterpret_cast<const __half2*>(&w0));
            const float2 h1 = __half22float2(*reinterpret_cast<const __half2*>(&w1));
            v = fma2(ph, pack2(h0.y, h1.y), pack2(h0.x, h1.x));
          }
        }
        if constexpr (WGT != 0) v = mul2(pack2(ww[2 * x], ww[2 * x + 1]), v);
        acc[x] = fma2(mm, v, acc[x]);
      }
    };
    // one step: the sensors j, j + 1 in the slots of `buf`, their offsets in u;
    // the next step's offsets into nu, the windows of the step after that
    auto step = [&](int j, const float4 (&u)[2], float4 (&nu)[2], int buf) {
      load_u(j + 2, nu);
      cp_async_wait<1>();
      __syncwarp();
      const uint4 q = lds_u4(bm_s + uint32_t(j) * 8u);  // sensors j and j + 1
      sensor(j, u[0], 2 * buf, __uint_as_float(q.y));
      sensor(j + 1, u[1], 2 * buf + 1, __uint_as_float(q.w));
      __syncwarp();  // every lane has read the slots before they are refilled
      issue(j + 4, buf);
    };
    for (int j = 0; j < nj; j += 4) {
      step(j, ua, ub, 0);
      if (j + 2 < nj) step(j + 2, ub, ua, 1);
    }
    cp_async_wait<0>();
    float r[4];
    unpack2(acc[0], r[0], r[1]);
    unpack2(acc[1], r[2], r[3]);
    *reinterpret_cast<float4*>(&ssum[sp][px0]) = make_float4(r[0], r[1], r[2], r[3]);
    __syncthreads();
    for (int q = threadIdx.x; q < P; q += 128) {
      float v = 0.0f;
#pragma unroll
      for (int ph = 0; ph < SW; ++ph) v += ssum[ph][q];
      if (final) {
        const int o = __ldcg(p.slot + int64_t(tile) * P + q);
        if (o >= 0) p.out[o] = v;
      } else {
        p.part[(int64_t(tile) * p.n_seg + seg) * P + q] = v;
      }
    }
    __syncthreads();
  }
}

template <typename K>
cudaError_t launch_pdl(K kern, unsigned grid, unsigned threads, const DirectParams& dp, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1u, 1u);
  cfg.blockDim = dim3(threads, 1u, 1u);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, dp);
}

constexpr int kMaxDevices = 64;

// Resident CTAs per SM of one kernel, looked up once per device (devices of a
// process may differ).
struct PerDevice {
  int per_sm[kMaxDevices] = {};
};

template <int P, int SW, int FMT, int DELAYS, int WGT>
cudaError_t launch_direct_fmt(const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  auto kern = gather_direct_kernel<P, SW, FMT, DELAYS, WGT>;
  const int threads = 32 * (P / 128) * SW;
  static PerDevice cache;  // resident CTAs per SM, per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (cache.per_sm[dev] == 0) {
    int v = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, threads, 0);
    if (e != cudaSuccess) return e;
    cache.per_sm[dev] = v > 0 ? v : 1;
  }
  const int64_t n_units = int64_t(dp.n_tiles) * dp.n_seg;
  const unsigned grid = unsigned(std::min<int64_t>(n_units, int64_t(cache.per_sm[dev]) * n_sm));
  e = launch_pdl(kern, grid, unsigned(threads), dp, st);
  if (e != cudaSuccess || !reduce) return e;
  const int64_t n = int64_t(dp.n_tiles) * P;
  const unsigned rgrid = unsigned(std::min<int64_t>((n + 255) / 256, int64_t(n_sm) * 8));
  return launch_pdl(direct_reduce_kernel<P, SW>, std::max(rgrid, 1u), 256u, dp, st);
}

template <int P, int SW, int FMT, int WB, int DELAYS, int WGT>
cudaError_t launch_window_fmt(const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  auto kern = gather_window_kernel<P, SW, FMT, WB, DELAYS, WGT>;
  static PerDevice cache;  // resident CTAs per SM, per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  if (cache.per_sm[dev] == 0) {
    int v = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kern, 128, 0);
    if (e != cudaSuccess) return e;
    cache.per_sm[dev] = v > 0 ? v : 1;
  }
  const int64_t n_units = int64_t(dp.n_tiles) * dp.n_seg;
  const unsigned grid = unsigned(std::min<int64_t>(n_units, int64_t(cache.per_sm[dev]) * n_sm));
  e = launch_pdl(kern, grid, 128u, dp, st);
  if (e != cudaSuccess || !reduce || dp.n_seg == 1) return e;  // one segment: the gather wrote the image
  const int64_t n = int64_t(dp.n_tiles) * P;
  const unsigned rgrid = unsigned(std::min<int64_t>((n + 255) / 256, int64_t(n_sm) * 8));
  return launch_pdl(direct_reduce_kernel<P, 1>, std::max(rgrid, 1u), 256u, dp, st);
}

template <int P, int SW, int WB, int DELAYS, int WGT>
cudaError_t launch_window_w(int fmt, const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  if (fmt == kBF32) return launch_window_fmt<P, SW, kBF32, WB, DELAYS, WGT>(dp, n_sm, st, reduce);
  if (fmt == kBBF16P) return launch_window_fmt<P, SW, kBBF16P, WB, DELAYS, WGT>(dp, n_sm, st, reduce);
  if (fmt == kBF16P) return launch_window_fmt<P, SW, kBF16P, WB, DELAYS, WGT>(dp, n_sm, st, reduce);
  return cudaErrorInvalidValue;
}

// The smallest slot (128, 192, 288 or 384 rows) that holds every window.
template <int P, int SW, int DELAYS, int WGT>
cudaError_t launch_window(int fmt, const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  if constexpr (DELAYS == 0 || P == 128) {
    if (dp.W <= 128) return launch_window_w<P, SW, 128, DELAYS, WGT>(fmt, dp, n_sm, st, reduce);
    if (dp.W <= 192) return launch_window_w<P, SW, 192, DELAYS, WGT>(fmt, dp, n_sm, st, reduce);
  }
  if constexpr (DELAYS == 0 && WGT == 0)
    if (dp.W > 288) return launch_window_w<P, SW, kWindowMaxRows, 0, 0>(fmt, dp, n_sm, st, reduce);
  if constexpr (DELAYS == 0) return launch_window_w<P, SW, 288, DELAYS, WGT>(fmt, dp, n_sm, st, reduce);
  return cudaErrorInvalidValue;
}

template <int P, int SW>
cudaError_t launch_window_mode(bool delays, int fmt, const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  if (dp.wanchor)
    return delays ? launch_window<P, SW, 1, 1>(fmt, dp, n_sm, st, reduce)
                  : launch_window<P, SW, 0, 1>(fmt, dp, n_sm, st, reduce);
  return delays ? launch_window<P, SW, 1, 0>(fmt, dp, n_sm, st, reduce)
                : launch_window<P, SW, 0, 0>(fmt, dp, n_sm, st, reduce);
}

template <int P, int SW, int DELAYS, int WGT>
cudaError_t launch_direct_w(int fmt, const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  if (fmt == kBF32) return launch_direct_fmt<P, SW, kBF32, DELAYS, WGT>(dp, n_sm, st, reduce);
  if (fmt == kBBF16P) return launch_direct_fmt<P, SW, kBBF16P, DELAYS, WGT>(dp, n_sm, st, reduce);
  if (fmt == kBF16P) return launch_direct_fmt<P, SW, kBF16P, DELAYS, WGT>(dp, n_sm, st, reduce);
  return cudaErrorInvalidValue;
}

template <int P, int SW, int DELAYS>
cudaError_t launch_direct_t(int fmt, const DirectParams& dp, int n_sm, cudaStream_t st, bool reduce) {
  return dp.wanchor ? launch_direct_w<P, SW, DELAYS, 1>(fmt, dp, n_sm, st, reduce)
                    : launch_direct_w<P, SW, DELAYS, 0>(fmt, dp, n_sm, st, reduce);
}

}  // namespace

size_t direct_part_floats(const GatherConfig& c, int n_tiles, int n_seg) {
  return size_t(n_tiles) * n_seg * c.SW * c.P;
}

cudaError_t launch_gather_direct(const GatherConfig& c, int fmt, const InstDesc& d, int n_sm,
                                 int* status, int* host_status, uint64_t timeout_ns,
                                 cudaStream_t st, bool reduce) {
  if (d.n_frames != 1 || c.FB != 1 || d.n_fg != 1 || n_sm < 1 || !d.part) return cudaErrorInvalidValue;
  DirectParams dp;
  dp.u = d.u;
  dp.anchor = d.anchor;
  dp.pix = d.pix;
  dp.wanchor = d.wanchor;
  dp.base = d.base;
  dp.slot = d.slot;
  dp.zero_runs = d.zero_runs;
  dp.b = d.b;
  dp.m = d.m;
  dp.out = d.out;
  dp.part = d.part;
  dp.status = status;
  dp.host_status = host_status;
  dp.timeout_ns = timeout_ns;
  dp.n_zero_runs = d.n_zero_runs;
  dp.n_sensors = d.n_sensors;
  dp.n_sensors_pad = d.n_sensors_pad;
  dp.n_t_pad = d.n_t_pad;
  dp.n_tiles = d.n_tiles;
  dp.n_seg = d.n_seg;
  dp.G = d.G;
  dp.W = d.W;
  const bool window = !c.no_window && dp.G <= 64 &&
                      window_pays(c.delays != 0, dp.wanchor != nullptr, c.P, dp.W,
                                  int64_t(dp.n_tiles) * dp.n_seg, dp.n_seg, n_sm);
  if (window && c.P == 128 && c.SW == 4) return launch_window_mode<128, 4>(c.delays != 0, fmt, dp, n_sm, st, reduce);
  if (window && c.P == 256 && c.SW == 2) return launch_window_mode<256, 2>(c.delays != 0, fmt, dp, n_sm, st, reduce);
  if (c.P == 128 && c.SW == 4)
    return c.delays ? launch_direct_t<128, 4, 1>(fmt, dp, n_sm, st, reduce)
                    : launch_direct_t<128, 4, 0>(fmt, dp, n_sm, st, reduce);
  if (c.P == 256 && c.SW == 2)
    return c.delays ? launch_direct_t<256, 2, 1>(fmt, dp, n_sm, st, reduce)
                    : launch_direct_t<256, 2, 0>(fmt, dp, n_sm, st, reduce);
  return cudaErrorInvalidValue;
}

}  // namespace patbp
