// kernels.cu -- sm_103a kernels of the on-line back projection (Eq. (BP)).
//
//   preprocess_kernel  b_k = 2 p_k - 2 t_k dp/dt|_k per (frame, sensor) row,
//                      t_k = k dt, central difference inside and one-sided
//                      differences at the ends; optional 16-bit (value, slope)
//                      pairs with a per-row scale.  Since t_k / dt = k the
//                      interior value is 2 p_k - k (p_{k+1} - p_{k-1}).
//   gather_kernel      out[f][r] = sum_s w_s * b_{f,s}(T_s(r)/dt) with linear
//                      interpolation (Sec. II-C) for units of 1 or 2 frames,
//                      defined in gather.cuh; this unit instantiates it for
//                      delays from the stored fast-marching table and holds
//                      the launchers of every gather (gather_rows.cuh: units
//                      of 4 to 32 frames).
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <cstdio>

#include "gather_rows.cuh"

namespace patbp {
// ---------------------------------------------------------- preprocessing --
template <int DT>
__device__ __forceinline__ float load_sample(const void* sig, int64_t i) {
  if constexpr (DT == 0) {
    return __ldg(static_cast<const float*>(sig) + i);
  } else if constexpr (DT == 1) {
    return __bfloat162float(static_cast<const __nv_bfloat16*>(sig)[i]);
  } else {
    return __half2float(static_cast<const __half*>(sig)[i]);
  }
}

// p_k0 .. p_{k0+7} of a row, times sc, zero outside [0, n): one or two 16-byte
// loads when the run lies in the row and is aligned (so signals read in place
// from host memory cost few requests), else one load per sample.
template <int DT>
__device__ __forceinline__ void load_run8(const void* sig, int64_t row0, int k0, int n, float sc,
                                          float* v) {
  const size_t esz = DT == 0 ? 4 : 2;
  const unsigned char* ptr = static_cast<const unsigned char*>(sig) + (row0 + k0) * int64_t(esz);
  if (k0 >= 0 && k0 + 8 <= n && (reinterpret_cast<uintptr_t>(ptr) & 15) == 0) {
    if constexpr (DT == 0) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(ptr));
      const float4 b = __ldg(reinterpret_cast<const float4*>(ptr) + 1);
      const float x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __fmul_rn(x[j], sc);
    } else {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(ptr));
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const unsigned short h = (unsigned short)(w[j >> 1] >> ((j & 1) * 16));
        const float x = DT == 1 ? __bfloat162float(__ushort_as_bfloat16(h)) : __half2float(__ushort_as_half(h));
        v[j] = __fmul_rn(x, sc);
      }
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = k0 + j;
      v[j] = (k >= 0 && k < n) ? __fmul_rn(load_sample<DT>(sig, row0 + k), sc) : 0.0f;
    }
  }
}

// The 16-bit (value, slope) pair of b_k and b_{k+1} scaled by inv: every
// product and difference is explicitly rounded, so the codes do not depend on
// how the compiler contracts the expression in the kernel that calls this.
template <int FMT>
__device__ __forceinline__ uint32_t encode_pair(float b0, float b1, float inv) {
  const float v0 = __fmul_rn(b0, inv), v1 = __fmul_rn(b1, inv);
  if constexpr (FMT == kBBF16P) {
    const __nv_bfloat16 q0 = __float2bfloat16_rn(v0);
    const __nv_bfloat16 q1 = __float2bfloat16_rn(__fsub_rn(v1, __bfloat162float(q0)));
    return uint32_t(__bfloat16_as_ushort(q0)) | (uint32_t(__bfloat16_as_ushort(q1)) << 16);
  } else {
    const __half q0 = __float2half_rn(v0);
    const __half q1 = __float2half_rn(__fsub_rn(v1, __half2float(q0)));
    return uint32_t(__half_as_ushort(q0)) | (uint32_t(__half_as_ushort(q1)) << 16);
  }
}

template <int N>
__device__ __forceinline__ void store_words(uint32_t* dst, const uint32_t (&w)[N]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N; i += 4)
      *reinterpret_cast<uint4*>(dst + i) = make_uint4(w[i], w[i + 1], w[i + 2], w[i + 3]);
  } else if constexpr (N == 2) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
  } else {
    dst[0] = w[0];
  }
}

// One CTA per (sensor, frame group) row; every thread owns K consecutive
// samples of the row for all FB frames and issues all its loads before any
// use; the samples just outside its run (p_{k0-1}, p_{k0+K}, p_{k0+K+1}) come
// from the neighbouring lanes by shuffles, so the loops run warp-uniformly.
// Rows are written frame-interleaved, K * FB words per thread.
template <int DT, int FMT, int FB>
__device__ __forceinline__ void preprocess_row(const PreParams& p, int s, int g) {
  constexpr int K = 8;
  __shared__ float red[8][FB];
  const int f0 = g * FB;
  const int fb_eff = min(FB, p.n_frames - f0);
  const int n = p.n_t;
  int64_t row0[FB];
  float sc[FB];
#pragma unroll
  for (int fb = 0; fb < FB; ++fb) {
    const int f = min(f0 + fb, p.n_frames - 1);
    const int64_t r = int64_t(f) * p.n_sensors + s;
    row0[fb] = r * n;
    sc[fb] = p.scales ? p.scales[r] : 1.0f;
  }
  // b_{k0..k0+K} of frame fb (K + 1 values; the last feeds the pair slope).
  // Products and differences are explicitly rounded (no contraction into
  // FMAs): the values do not depend on how the compiler schedules them.  All
  // lanes of a warp call it together (consecutive runs, k0 = lane K + ...).
  const int lane = threadIdx.x & 31;
  auto sample = [&](int fb, int k) {
    return (k >= 0 && k < n) ? __fmul_rn(load_sample<DT>(p.sig, row0[fb] + k), sc[fb]) : 0.0f;
  };
  auto b_run = [&](int fb, int k0, float (&b)[K + 1]) {
    static_assert(K == 8, "runs of 8 samples");
    float v[K + 3];  // p_{k0-1} .. p_{k0+K+1}
    load_run8<DT>(p.sig, row0[fb], k0, n, sc[fb], v + 1);
    const float prev = __shfl_up_sync(0xffffffffu, v[K], 1);
    const float nx1 = __shfl_down_sync(0xffffffffu, v[1], 1);
    const float nx2 = __shfl_down_sync(0xffffffffu, v[2], 1);
    v[0] = lane == 0 ? sample(fb, k0 - 1) : prev;
    v[K + 1] = lane == 31 ? sample(fb, k0 + K) : nx1;
    v[K + 2] = lane == 31 ? sample(fb, k0 + K + 1) : nx2;
#pragma unroll
    for (int j = 0; j <= K; ++j) {
      const int k = k0 + j;
      float r;
      if (k >= n) r = 0.0f;
      else if (k == 0) r = 2.0f * v[j + 1];
      else if (k == n - 1) r = fmaf(-2.0f * float(k), __fsub_rn(v[j + 1], v[j]), 2.0f * v[j + 1]);
      else r = fmaf(-float(k), __fsub_rn(v[j + 2], v[j]), 2.0f * v[j + 1]);
      b[j] = r;
    }
  };
  float inv[FB], sigma[FB];
#pragma unroll
  for (int fb = 0; fb < FB; ++fb) sigma[fb] = inv[fb] = 1.0f;
  if constexpr (FMT != kBF32) {
    float mx[FB];
#pragma unroll
    for (int fb = 0; fb < FB; ++fb) mx[fb] = 0.0f;
    for (int kw = (threadIdx.x & ~31) * K; kw < n; kw += blockDim.x * K) {
      const int k0 = kw + lane * K;  // runs past the row give b = 0
#pragma unroll
      for (int fb = 0; fb < FB; ++fb) {
        float b[K + 1];
        b_run(fb, k0, b);
#pragma unroll
        for (int j = 0; j < K; ++j) mx[fb] = fmaxf(mx[fb], fabsf(b[j]));
      }
    }
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
#pragma unroll
    for (int fb = 0; fb < FB; ++fb) {
      float v = mx[fb];
      for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
      if (l == 0) red[w][fb] = v;
    }
    __syncthreads();
#pragma unroll
    for (int fb = 0; fb < FB; ++fb) {
      float v = 0.0f;
      for (int q = 0; q < int(blockDim.x >> 5); ++q) v = fmaxf(v, red[q][fb]);
      sigma[fb] = v > 0.0f ? v : 1.0f;
      inv[fb] = 1.0f / sigma[fb];
    }
  }
  uint32_t* dst = static_cast<uint32_t*>(p.b) + (int64_t(g) * p.n_sensors + s) * p.n_t_pad * FB;
  for (int kw = (threadIdx.x & ~31) * K; kw < p.n_t_pad; kw += blockDim.x * K) {
    const int k0 = kw + lane * K;
    uint32_t w[K * FB];
#pragma unroll
    for (int fb = 0; fb < FB; ++fb) {
      if (fb < fb_eff) {
        float b[K + 1];
        b_run(fb, k0, b);
#pragma unroll
        for (int j = 0; j < K; ++j) {
          if constexpr (FMT == kBF32) w[j * FB + fb] = __float_as_uint(b[j]);
          else w[j * FB + fb] = encode_pair<FMT>(b[j], b[j + 1], inv[fb]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < K; ++j) w[j * FB + fb] = 0u;
      }
    }
    if (k0 < p.n_t_pad) store_words<K * FB>(dst + int64_t(k0) * FB, w);
  }
  if (threadIdx.x < FB) {
    const int fb = threadIdx.x;
    float mval = 0.0f;
#pragma unroll
    for (int q = 0; q < FB; ++q)
      if (q == fb && fb < fb_eff) mval = p.weights[s] * sigma[q];
    p.m[(int64_t(g) * p.n_sensors_pad + s) * FB + fb] = mval;
  }
}

// The same rows for FB >= 2 frames per group, laid out for occupancy: thread
// t works on frame t mod FB and runs of 8 samples, frames fastest across the
// lanes, so a run's neighbouring runs of the same frame sit FB lanes away
// (shuffles by FB), every store instruction writes whole 32-byte pieces of
// FB * 8 consecutive words, and a thread keeps 11 samples instead of FB x 11.
// Each sample is the same expression as in preprocess_row, so the integrand
// has the same bits whatever the frames per group.
template <int DT, int FMT, int FB>
__device__ __forceinline__ void preprocess_row_frames(const PreParams& p, int s, int g) {
  static_assert(FB >= 2 && FB <= 4 && (FB & (FB - 1)) == 0, "frames per group");
  constexpr int K = 8;
  constexpr int RUNS = 256 / FB;  // runs of one frame per block pass
  __shared__ float red[8][FB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int fb = threadIdx.x & (FB - 1);
  const int run = threadIdx.x / FB;
  const int f0 = g * FB;
  const int fb_eff = min(FB, p.n_frames - f0);
  const int n = p.n_t;
  const int f = min(f0 + fb, p.n_frames - 1);
  const int64_t r = int64_t(f) * p.n_sensors + s;
  const int64_t row0 = r * n;
  const float sc = p.scales ? p.scales[r] : 1.0f;
  auto sample = [&](int k) {
    return (k >= 0 && k < n) ? __fmul_rn(load_sample<DT>(p.sig, row0 + k), sc) : 0.0f;
  };
  // b_{k0..k0+K} of this thread's frame; all lanes of a warp call it together
  auto b_run = [&](int k0, float (&b)[K + 1]) {
    float v[K + 3];  // p_{k0-1} .. p_{k0+K+1}
    load_run8<DT>(p.sig, row0, k0, n, sc, v + 1);
    const float prev = __shfl_up_sync(0xffffffffu, v[K], FB);
    const float nx1 = __shfl_down_sync(0xffffffffu, v[1], FB);
    const float nx2 = __shfl_down_sync(0xffffffffu, v[2], FB);
    v[0] = lane < FB ? sample(k0 - 1) : prev;
    v[K + 1] = lane >= 32 - FB ? sample(k0 + K) : nx1;
    v[K + 2] = lane >= 32 - FB ? sample(k0 + K + 1) : nx2;
#pragma unroll
    for (int j = 0; j <= K; ++j) {
      const int k = k0 + j;
      float x;
      if (k >= n) x = 0.0f;
      else if (k == 0) x = 2.0f * v[j + 1];
      else if (k == n - 1) x = fmaf(-2.0f * float(k), __fsub_rn(v[j + 1], v[j]), 2.0f * v[j + 1]);
      else x = fmaf(-float(k), __fsub_rn(v[j + 2], v[j]), 2.0f * v[j + 1]);
      b[j] = x;
    }
  };
  float sigma = 1.0f, inv = 1.0f;
  if constexpr (FMT != kBF32) {
    float mx = 0.0f;
    for (int kw = 0; kw < n; kw += RUNS * K) {
      const int k0 = kw + run * K;  // runs past the row give b = 0
      float b[K + 1];
      b_run(k0, b);
#pragma unroll
      for (int j = 0; j < K; ++j) mx = fmaxf(mx, fabsf(b[j]));
    }
    for (int o = FB; o < 32; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane < FB) red[warp][lane] = mx;
    __syncthreads();
    float v = 0.0f;
    for (int q = 0; q < int(blockDim.x >> 5); ++q) v = fmaxf(v, red[q][fb]);
    sigma = v > 0.0f ? v : 1.0f;
    inv = 1.0f / sigma;
  }
  uint32_t* dst = static_cast<uint32_t*>(p.b) + (int64_t(g) * p.n_sensors + s) * p.n_t_pad * FB;
  const bool live = fb < fb_eff;
  for (int kw = 0; kw < p.n_t_pad; kw += RUNS * K) {
    const int k0 = kw + run * K;
    float b[K + 1];
    b_run(k0, b);
    if (k0 >= p.n_t_pad) continue;
#pragma unroll
    for (int j = 0; j < K; ++j) {
      uint32_t wv = 0u;
      if (live) {
        if constexpr (FMT == kBF32) wv = __float_as_uint(b[j]);
        else wv = encode_pair<FMT>(b[j], b[j + 1], inv);
      }
      dst[int64_t(k0 + j) * FB + fb] = wv;
    }
  }
  if (threadIdx.x < FB) p.m[(int64_t(g) * p.n_sensors_pad + s) * FB + fb] = live ? p.weights[s] * sigma : 0.0f;
}

// Eq. (BP) integrand b_k of one row of n samples from p_{k-1}, p_k, p_{k+1}
// (explicitly rounded, the expression of the two layouts above).
__device__ __forceinline__ float integrand(int k, int n, float pm, float p0, float p1) {
  if (k >= n) return 0.0f;
  if (k == 0) return 2.0f * p0;
  if (k == n - 1) return fmaf(-2.0f * float(k), __fsub_rn(p0, pm), 2.0f * p0);
  return fmaf(-float(k), __fsub_rn(p1, pm), 2.0f * p0);
}

// Two 16-bit samples of a word as FP32 (low half first).
template <int DT>
__device__ __forceinline__ float2 unpack_samples(uint32_t w) {
  if constexpr (DT == 1) return make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u));
  else return __half22float2(*reinterpret_cast<const __half2*>(&w));
}

// Codes of samples k0 .. k0 + 7 of a 16-bit row, zero outside [0, n).
__device__ __forceinline__ uint4 load_codes8(const uint16_t* row, int k0, int n) {
  const uint16_t* ptr = row + k0;
  if (k0 >= 0 && k0 + 8 <= n && (reinterpret_cast<uintptr_t>(ptr) & 15) == 0)
    return __ldg(reinterpret_cast<const uint4*>(ptr));
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = k0 + 2 * j;
    const uint32_t lo = k >= 0 && k < n ? __ldg(row + k) : 0u, hi = k + 1 >= 0 && k + 1 < n ? __ldg(row + k + 1) : 0u;
    w[j] = lo | hi << 16;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Rows of 8, 16 or 32 frames per group.  A row of FB frames is contiguous, so
// frames must be fastest across the lanes for the stores while the signals are
// contiguous in time: chunks of KC samples of all frames go through shared
// memory (odd pitches keep both sides nearly free of bank conflicts), the next
// chunk's loads in flight while one is computed.  Bound by HBM for FP32 (64
// paper-shaped frames: 538 MB); by instruction issue for 16-bit signals, whose
// integrands need the row's largest |b| first: a pass over the signals with a
// warp per frame (the second pass finds them in L2).  part of parts: the share
// of the row's chunks that this CTA writes (short launches split rows to fill
// the chip; each share repeats the first pass).
template <int DT, int FMT, int FB>
__device__ __forceinline__ void preprocess_row_tiles(const PreParams& p, int s, int g, int part, int parts) {
  static_assert(FB == 8 || FB == 16 || FB == 32, "frames per group");
  constexpr int KC = 4096 / FB, COLS = KC + 4;            // samples c0 - 2 .. c0 + KC + 1
  constexpr int W = DT == 0 ? 1 : 2;                      // samples of one word
  constexpr int WORDS = COLS / W, PITCH = WORDS + 1;      // odd
  constexpr int RUNS = 256 / FB, RUN = KC / RUNS;         // 16 samples per thread and chunk
  constexpr int NF = FB / 8;                              // frames of a warp
  constexpr int NL = (WORDS + 31) / 32;                   // loads per frame and lane
  __shared__ uint32_t tile[FB][PITCH];
  __shared__ float sig_s[FB];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int f0 = g * FB, live = min(FB, p.n_frames - f0), n = p.n_t;
  const int fb = threadIdx.x & (FB - 1), run = threadIdx.x / FB;
  int64_t row0[NF];
#pragma unroll
  for (int i = 0; i < NF; ++i) row0[i] = (int64_t(f0 + min(warp + 8 * i, live - 1)) * p.n_sensors + s) * n;
  const float sc = p.scales && fb < live ? p.scales[int64_t(f0 + fb) * p.n_sensors + s] : 1.0f;
  float sigma = 1.0f, inv = 1.0f;
  if constexpr (FMT != kBF32) {
    // largest |b| per frame: 8 samples per lane and step, UN steps in flight
    constexpr int UN = 4 / NF;
    float mx[NF], scf[NF];
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      mx[i] = 0.0f;
      scf[i] = p.scales ? p.scales[row0[i] / n] : 1.0f;
    }
    for (int kw = 0; kw < n; kw += 256 * UN) {
      uint4 raw[UN][NF];
      uint32_t edge[UN][NF];  // the sample before lane 0's, after lane 31's
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          const uint16_t* row = static_cast<const uint16_t*>(p.sig) + row0[i];
          const int k0 = kw + u * 256 + lane * 8, ke = lane == 0 ? k0 - 1 : k0 + 8;
          raw[u][i] = load_codes8(row, k0, n);
          edge[u][i] = (lane == 0 || lane == 31) && ke >= 0 && ke < n ? __ldg(row + ke) : 0u;
        }
#pragma unroll
      for (int u = 0; u < UN; ++u)
#pragma unroll
        for (int i = 0; i < NF; ++i) {
          const int k0 = kw + u * 256 + lane * 8;
          const uint32_t w[4] = {raw[u][i].x, raw[u][i].y, raw[u][i].z, raw[u][i].w};
          float v[10];  // p_{k0-1} .. p_{k0+8}
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float2 x = unpack_samples<DT>(w[j]);
            v[1 + 2 * j] = __fmul_rn(x.x, scf[i]);
            v[2 + 2 * j] = __fmul_rn(x.y, scf[i]);
          }
          const float e = __fmul_rn(unpack_samples<DT>(edge[u][i]).x, scf[i]);
          const float prev = __shfl_up_sync(0xffffffffu, v[8], 1), nxt = __shfl_down_sync(0xffffffffu, v[1], 1);
          v[0] = lane == 0 ? e : prev;
          v[9] = lane == 31 ? e : nxt;
          if (k0 > 0 && k0 + 8 < n) {
            const float kf = -float(k0);
#pragma unroll
            for (int j = 0; j < 8; ++j)
              mx[i] = fmaxf(mx[i], fabsf(fmaf(kf - float(j), __fsub_rn(v[j + 2], v[j]), 2.0f * v[j + 1])));
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) mx[i] = fmaxf(mx[i], fabsf(integrand(k0 + j, n, v[j], v[j + 1], v[j + 2])));
          }
        }
    }
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      for (int o = 16; o > 0; o >>= 1) mx[i] = fmaxf(mx[i], __shfl_xor_sync(0xffffffffu, mx[i], o));
      if (lane == 0) sig_s[warp + 8 * i] = mx[i] > 0.0f ? mx[i] : 1.0f;
    }
    __syncthreads();
    sigma = sig_s[fb];
    inv = 1.0f / sigma;
  }
  // 16-bit signals go two samples per load when every row starts on 4 bytes
  const bool pairs = W == 2 && (n & 1) == 0 && (reinterpret_cast<uintptr_t>(p.sig) & 3) == 0;
  uint32_t raw[NF][NL];
  auto fetch = [&](int c0) {
    const bool whole = c0 > 0 && c0 + KC + 2 <= n && (W == 1 || pairs);
#pragma unroll
    for (int i = 0; i < NF; ++i) {
      const bool on = warp + 8 * i < live;  // absent frames are stored as zeros
#pragma unroll
      for (int l = 0; l < NL; ++l) {
        const int q = l * 32 + lane, k = c0 - 2 + W * q;
        uint32_t w = 0u;
        if constexpr (DT == 0) {
          const float* src = static_cast<const float*>(p.sig) + row0[i] + k;
          if (on && q < WORDS && (whole || (k >= 0 && k < n))) w = __float_as_uint(__ldg(src));
        } else {
          const uint16_t* src = static_cast<const uint16_t*>(p.sig) + row0[i] + k;
          if (whole) {
            if (on && q < WORDS) w = __ldg(reinterpret_cast<const uint32_t*>(src));
          } else if (on && q < WORDS && k >= 0 && k < n) {
            if (pairs) w = __ldg(reinterpret_cast<const uint32_t*>(src));
            else w = uint32_t(__ldg(src)) | (k + 1 < n ? uint32_t(__ldg(src + 1)) << 16 : 0u);
          }
        }
        raw[i][l] = w;
      }
    }
  };
  uint32_t* dst = static_cast<uint32_t*>(p.b) + (int64_t(g) * p.n_sensors + s) * p.n_t_pad * FB + fb;
  const int chunks = (p.n_t_pad + KC - 1) / KC;
  const int cb = int(int64_t(chunks) * part / parts) * KC, ce = int(int64_t(chunks) * (part + 1) / parts) * KC;
  if (cb < ce) fetch(cb);
  for (int c0 = cb; c0 < ce; c0 += KC) {
    if (c0 != cb) __syncthreads();  // the chunk before has been read
#pragma unroll
    for (int i = 0; i < NF; ++i)
#pragma unroll
      for (int l = 0; l < NL; ++l)
        if (l * 32 + lane < WORDS) tile[warp + 8 * i][l * 32 + lane] = raw[i][l];
    __syncthreads();
    if (c0 + KC < ce) fetch(c0 + KC);
    const uint32_t* row = tile[fb] + run * RUN / W;  // the word of p_{k0-2}
    const int k0 = c0 + run * RUN;
    if (k0 >= p.n_t_pad) continue;
    uint32_t* out = dst + int64_t(k0) * FB;
    // p_{k0-1}, p_{k0}, p_{k0+1}, then p_{k+2} for k = k0, k0 + 1, ..
    float pm, pc, pn, later = 0.0f;
    if constexpr (W == 1) {
      pm = __fmul_rn(__uint_as_float(row[1]), sc);
      pc = __fmul_rn(__uint_as_float(row[2]), sc);
      pn = __fmul_rn(__uint_as_float(row[3]), sc);
    } else {
      const float2 x = unpack_samples<DT>(row[0]), y = unpack_samples<DT>(row[1]);
      pm = __fmul_rn(x.y, sc);
      pc = __fmul_rn(y.x, sc);
      pn = __fmul_rn(y.y, sc);
    }
    auto ahead = [&](int j) {  // p_{k0 + j + 2}
      if constexpr (W == 1) return __fmul_rn(__uint_as_float(row[j + 4]), sc);
      if (j & 1) return later;
      const float2 x = unpack_samples<DT>(row[j / 2 + 2]);
      later = __fmul_rn(x.y, sc);
      return __fmul_rn(x.x, sc);
    };
    if (k0 > 0 && k0 + RUN + 1 < n) {  // inside the record: one expression
      float kf = -float(k0);
      float b = fmaf(kf, __fsub_rn(pn, pm), 2.0f * pc);
#pragma unroll
      for (int j = 0; j < RUN; ++j) {
        const float pn2 = ahead(j);
        const float b1 = fmaf(kf - float(j + 1), __fsub_rn(pn2, pc), 2.0f * pn);
        if constexpr (FMT == kBF32) out[j * FB] = __float_as_uint(b);
        else out[j * FB] = encode_pair<FMT>(b, b1, inv);
        b = b1;
        pc = pn;
        pn = pn2;
      }
    } else {
      float b = integrand(k0, n, pm, pc, pn);
#pragma unroll
      for (int j = 0; j < RUN; ++j) {
        const float pn2 = ahead(j);
        const float b1 = integrand(k0 + j + 1, n, pc, pn, pn2);
        uint32_t wv;
        if constexpr (FMT == kBF32) wv = __float_as_uint(b);
        else wv = encode_pair<FMT>(b, b1, inv);
        if (k0 + j < p.n_t_pad) out[j * FB] = wv;
        b = b1;
        pc = pn;
        pn = pn2;
      }
    }
  }
  if (part == 0 && threadIdx.x < FB)
    p.m[(int64_t(g) * p.n_sensors_pad + s) * FB + fb] = fb < live ? p.weights[s] * sigma : 0.0f;
}

// One (sensor, frame group) row per CTA: the sample-run layout for single
// frames, the frame-fast one for 2 and 4, tiles for 8, 16 and 32.
template <int DT, int FMT, int FB>
__device__ __forceinline__ void preprocess_group(const PreParams& p, int s, int g, int part = 0,
                                                 int parts = 1) {
  if constexpr (FB == 1) preprocess_row<DT, FMT, FB>(p, s, g);
  else if constexpr (FB >= 8) preprocess_row_tiles<DT, FMT, FB>(p, s, g, part, parts);
  else preprocess_row_frames<DT, FMT, FB>(p, s, g);
}

template <int DT, int FMT, int FB>
__global__ void __launch_bounds__(256) preprocess_kernel(const PreParams p) {
  // let the gather that depends on this kernel start its prologue now (late: as
  // the CTAs exit)
  if (!p.late) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  preprocess_group<DT, FMT, FB>(p, blockIdx.x, blockIdx.y, blockIdx.z, gridDim.z);
}

// Several instances in one launch: CTA x belongs to the instance whose range
// [cta_begin[i], cta_begin[i+1]) holds it; inside it, (sensor, frame group).
template <int DT, int FMT, int FB>
__global__ void __launch_bounds__(256) preprocess_multi_kernel(const __grid_constant__ PreMultiParams p) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  int lo = 0, hi = p.n_inst - 1;
  const int64_t x = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (p.cta_begin[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  const PreParams& q = p.inst[lo];
  const int64_t loc = x - p.cta_begin[lo];
  preprocess_group<DT, FMT, FB>(q, int(loc % q.n_sensors), int(loc / q.n_sensors));
}


// ------------------------------------------------------------- wait probe --
__global__ void status_export_kernel(const int* status, int* host_status) { *host_status = *status; }

cudaError_t launch_status_export(const int* status, int* host_status, cudaStream_t st) {
  status_export_kernel<<<1, 1, 0, st>>>(status, host_status);
  return cudaGetLastError();
}

__global__ void wait_probe_kernel(int* status, uint64_t timeout_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  // nothing ever arrives on `bar`: the bounded wait must give up
  if (threadIdx.x == 0) {
    if (!mbar_wait_bounded(&bar, 0, timeout_ns, nullptr)) atomicOr(status, kStatusTimeout);
    // complete the phase ourselves so the barrier is left in a clean state
    mbar_arrive(&bar);
  }
}

// --------------------------------------------------------------- launchers --
size_t gather_smem_bytes(const GatherConfig& c, int Wst) {
  if (c.FB >= 4)  // the ring, two zero rows and the running sums
    return size_t(kRowsHeader) + c.ring + 2 * c.FB * 4 + (c.total ? size_t(c.P) * c.FB * 4 : 0);
  const StageLayout L(c.S, c.P, c.FB, Wst, c.delays | (c.wgt << 1));
  return size_t(kHeaderBytes) + kMetaBytes + L.bytes * c.stages + 2 * size_t(c.SW) * c.FB * c.P * 4;
}

template <int DT, int FMT>
static cudaError_t launch_pre_fb(const PreParams& p, cudaStream_t st) {
  dim3 grid(p.n_sensors, (p.n_frames + p.FB - 1) / p.FB);
  // tiles: rows are split in time while that fills the chip (4 CTAs per SM), but
  // not 16-bit rows in host memory, of which every share would read all twice
  // (16 BF16 frames of 128 sensors x 4 000 samples: 225 us in 2 shares, 125 whole);
  // FP32 rows there in half as many (32 frames of 64 sensors: 48 us in 2, 44 whole)
  if (p.FB >= 8 && !(DT != 0 && p.over_link)) {
    const int64_t chunks = (int64_t(p.n_t_pad) * p.FB + 4095) / 4096, rows = int64_t(grid.x) * grid.y;
    grid.z = unsigned(std::max<int64_t>(1, std::min<int64_t>(chunks, int64_t(p.over_link ? 2 : 4) * p.n_sm / rows)));
  }
  switch (p.FB) {
    case 1: preprocess_kernel<DT, FMT, 1><<<grid, 256, 0, st>>>(p); break;
    case 2: preprocess_kernel<DT, FMT, 2><<<grid, 256, 0, st>>>(p); break;
    case 4: preprocess_kernel<DT, FMT, 4><<<grid, 256, 0, st>>>(p); break;
    case 8: preprocess_kernel<DT, FMT, 8><<<grid, 256, 0, st>>>(p); break;
    case 16: preprocess_kernel<DT, FMT, 16><<<grid, 256, 0, st>>>(p); break;
    case 32: preprocess_kernel<DT, FMT, 32><<<grid, 256, 0, st>>>(p); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <int DT, int FMT>
static cudaError_t launch_pre_multi_fb(const PreMultiParams& p, cudaStream_t st) {
  const int64_t ctas = p.cta_begin[p.n_inst];
  if (ctas <= 0) return cudaSuccess;
  const dim3 grid(static_cast<unsigned>(ctas), 1u, 1u);
  switch (p.FB) {
    case 1: preprocess_multi_kernel<DT, FMT, 1><<<grid, 256, 0, st>>>(p); break;
    case 2: preprocess_multi_kernel<DT, FMT, 2><<<grid, 256, 0, st>>>(p); break;
    case 4: preprocess_multi_kernel<DT, FMT, 4><<<grid, 256, 0, st>>>(p); break;
    case 8: preprocess_multi_kernel<DT, FMT, 8><<<grid, 256, 0, st>>>(p); break;
    case 16: preprocess_multi_kernel<DT, FMT, 16><<<grid, 256, 0, st>>>(p); break;
    case 32: preprocess_multi_kernel<DT, FMT, 32><<<grid, 256, 0, st>>>(p); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_preprocess_multi(const PreMultiParams& p, cudaStream_t st) {
  if (p.n_inst < 1 || p.n_inst > kMaxInst) return cudaErrorInvalidValue;
  for (int i = 0; i < p.n_inst; ++i)
    if (p.inst[i].dtype != p.dtype || p.inst[i].fmt != p.fmt || p.inst[i].FB != p.FB)
      return cudaErrorInvalidValue;
  if (p.dtype == 0 && p.fmt == kBF32) return launch_pre_multi_fb<0, kBF32>(p, st);
  if (p.dtype == 1 && p.fmt == kBBF16P) return launch_pre_multi_fb<1, kBBF16P>(p, st);
  if (p.dtype == 2 && p.fmt == kBF16P) return launch_pre_multi_fb<2, kBF16P>(p, st);
  return cudaErrorInvalidValue;
}

const void* gather_kernel_func(const GatherConfig& c, int fmt);
const void* preprocess_multi_func(int dtype, int fmt, int FB);

cudaError_t launch_preprocess(const PreParams& p, cudaStream_t st) {
  if (p.dtype == 0 && p.fmt == kBF32) return launch_pre_fb<0, kBF32>(p, st);
  if (p.dtype == 1 && p.fmt == kBBF16P) return launch_pre_fb<1, kBBF16P>(p, st);
  if (p.dtype == 2 && p.fmt == kBF16P) return launch_pre_fb<2, kBF16P>(p, st);
  return cudaErrorInvalidValue;
}

static cudaError_t rows_dispatch(const GatherConfig& c, int fmt, const StreamParams* p, int grid,
                                 cudaStream_t st, int* resident, const void** func) {
  const size_t smem = p ? gather_smem_bytes(c, p->Wst) : 0;
  if (c.wgt)
    return c.delays ? rows_dispatch_3(c, fmt, p, smem, grid, st, resident, func)
                    : rows_dispatch_2(c, fmt, p, smem, grid, st, resident, func);
  return c.delays ? rows_dispatch_1(c, fmt, p, smem, grid, st, resident, func)
                  : rows_dispatch_0(c, fmt, p, smem, grid, st, resident, func);
}

size_t rows_group_bytes(const GatherConfig& c, int rows) {
  return RowsGroup(1, c.P, c.FB, c.delays | (c.wgt << 1)).bytes(rows, c.FB);
}

const void* rows_reduce_func(int FB) {
  switch (FB) {
    case 4: return reinterpret_cast<const void*>(rows_reduce_kernel<4>);
    case 8: return reinterpret_cast<const void*>(rows_reduce_kernel<8>);
    case 16: return reinterpret_cast<const void*>(rows_reduce_kernel<16>);
    case 32: return reinterpret_cast<const void*>(rows_reduce_kernel<32>);
  }
  return nullptr;
}

bool rows_needs_reduce(const StreamParams& p) {
  for (int i = 0; i < p.n_inst; ++i)
    if (p.split && p.inst[i].n_seg > 1) return true;
  return false;
}

template <int FB>
static cudaError_t launch_rows_reduce(const StreamParams& p, int P, int n_sm, cudaStream_t st) {
  int64_t n = 0;  // threads: one per pixel and 4 frames
  for (int i = 0; i < p.n_inst; ++i) n += int64_t(p.inst[i].n_fg) * p.inst[i].n_tiles * P * (FB / 4);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(std::min<int64_t>((n + 255) / 256, int64_t(n_sm) * 8)));
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, rows_reduce_kernel<FB>, p, P);
}

static cudaError_t launch_rows(const GatherConfig& c, int fmt, const StreamParams& p, int grid,
                               cudaStream_t st) {
  cudaError_t e = rows_dispatch(c, fmt, &p, grid, st, nullptr, nullptr);
  if (e != cudaSuccess || !rows_needs_reduce(p)) return e;
  switch (c.FB) {
    case 4: return launch_rows_reduce<4>(p, c.P, c.n_sm, st);
    case 8: return launch_rows_reduce<8>(p, c.P, c.n_sm, st);
    case 16: return launch_rows_reduce<16>(p, c.P, c.n_sm, st);
    case 32: return launch_rows_reduce<32>(p, c.P, c.n_sm, st);
  }
  return cudaErrorInvalidValue;
}

static cudaError_t gather_dispatch(const GatherConfig& c, int fmt, const StreamParams& p, int grid,
                                   cudaStream_t st, int* resident, int n_sm) {
  if (c.FB >= 4) return rows_dispatch(c, fmt, &p, grid, st, resident, nullptr);
  if (c.wgt)
    return c.delays ? gather_dispatch_wgt_const(c, fmt, p, grid, st, resident, n_sm)
                    : gather_dispatch_wgt(c, fmt, p, grid, st, resident, n_sm);
  if (c.delays) return gather_dispatch_const(c, fmt, p, grid, st, resident, n_sm);
  return gather_dispatch_t<0>(c, fmt, p, grid, st, resident, n_sm);
}

int gather_resident_ctas(const GatherConfig& c, int fmt, int Wst, int n_sm) {
  StreamParams dummy;
  dummy.Wst = Wst;
  int resident = 0;
  if (gather_dispatch(c, fmt, dummy, 0, nullptr, &resident, n_sm) != cudaSuccess) return 0;
  return resident;
}

cudaError_t launch_gather(const GatherConfig& c, int fmt, const StreamParams& p, int grid,
                          cudaStream_t st) {
  if (p.stages < 1 || p.stages > kMaxStages || p.S < 1 || (c.FB < 4 && (p.S % 4 || p.S % c.SW)) || p.S > kMaxS ||
      p.Wst % 8 || p.n_inst < 1 || p.n_inst > kMaxInst || grid < 1)
    return cudaErrorInvalidValue;
  for (int i = 0; i < p.n_inst; ++i)
    if ((c.FB >= 4 && p.inst[i].G > 64) || p.inst[i].G % p.S || p.inst[i].G > kMaxG || p.inst[i].Wst > p.Wst) return cudaErrorInvalidValue;
  if (p.n_units == 0) return cudaSuccess;
  if (c.direct) {
    // one frame after the other: frame f's integrand rows and multipliers are
    // frame group f of the one-frame-per-group layout; the phase sums are reused
    if (p.n_inst != 1 || c.FB != 1) return cudaErrorInvalidValue;
    const InstDesc& d = p.inst[0];
    const size_t word = 4;  // integrand words are 32-bit in every format
    for (int f = 0; f < d.n_frames; ++f) {
      InstDesc df = d;
      df.n_frames = 1;
      df.n_fg = 1;
      df.b = static_cast<const unsigned char*>(d.b) + size_t(f) * d.n_sensors * d.n_t_pad * word;
      df.m = d.m + size_t(f) * d.n_sensors_pad;
      df.out = d.out + int64_t(f) * d.out_stride;
      cudaError_t e = launch_gather_direct(c, fmt, df, c.n_sm, p.status, nullptr, p.timeout_ns, st);
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (c.FB >= 4) {
    // any sensor of the launch must fit the ring
    if (p.ring != c.ring || p.ring % 128 || p.S > kRowsMaxS || rows_group_bytes(c, p.Wst) > size_t(p.ring)) return cudaErrorInvalidValue;
    return launch_rows(c, fmt, p, grid, st);
  }
  return gather_dispatch(c, fmt, p, grid, st, nullptr, 0);
}

const void* gather_kernel_func(const GatherConfig& c, int fmt) {
  if (c.FB >= 4) {
    const void* f = nullptr;
    return rows_dispatch(c, fmt, nullptr, 0, nullptr, nullptr, &f) == cudaSuccess ? f : nullptr;
  }
  if (c.wgt) return c.delays ? gather_func_wgt_const(c, fmt) : gather_func_wgt(c, fmt);
  return c.delays ? gather_func_const(c, fmt) : gather_func_t<0>(c, fmt);
}

template <int DT, int FMT>
static const void* pre_multi_func_fb(int FB) {
  switch (FB) {
    case 1: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 1>);
    case 2: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 2>);
    case 4: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 4>);
    case 8: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 8>);
    case 16: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 16>);
    case 32: return reinterpret_cast<const void*>(preprocess_multi_kernel<DT, FMT, 32>);
  }
  return nullptr;
}

const void* preprocess_multi_func(int dtype, int fmt, int FB) {
  if (dtype == 0 && fmt == kBF32) return pre_multi_func_fb<0, kBF32>(FB);
  if (dtype == 1 && fmt == kBBF16P) return pre_multi_func_fb<1, kBBF16P>(FB);
  if (dtype == 2 && fmt == kBF16P) return pre_multi_func_fb<2, kBF16P>(FB);
  return nullptr;
}

cudaError_t launch_wait_probe(int* status, uint64_t timeout_ns, cudaStream_t st) {
  wait_probe_kernel<<<1, 32, 0, st>>>(status, timeout_ns);
  return cudaGetLastError();
}

}  // namespace patbp
