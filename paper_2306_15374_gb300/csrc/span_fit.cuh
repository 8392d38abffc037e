// Span fits of the variable partitioner (§3.1 Regressor over the spans of §3.2.2): the moments of a
// span's values by one thread or a group, and the residual range under a span's line.
//
// Moments of a span (w = the value as two's complement int64, x = the local index): T0 = sum w,
// T1 = sum x w, and min and max of w. The fit's least-squares moment is S = sum (2x - (N-1)) w =
// 2 T1 - (N-1) T0, and two adjacent spans' moments combine exactly (the right span's x shifts by
// the left span's length: T1 gains N_left T0_right).
#pragma once

#include "fit.cuh"
#include "leco_internal.cuh"

namespace leco {
namespace {

constexpr uint32_t kFull = 0xffffffffu;

struct SpanStats {
  i128 T0;
  i128 T1;
  int64_t mn;
  int64_t mx;
};

__device__ __forceinline__ SpanStats combine_stats(const SpanStats& l, uint64_t nl, const SpanStats& r) {
  SpanStats c;
  c.T0 = l.T0 + r.T0;
  c.T1 = l.T1 + r.T1 + mul_i128_u64(r.T0, nl);
  c.mn = min(l.mn, r.mn);
  c.mx = max(l.mx, r.mx);
  return c;
}

// the fit's least-squares moment of a span of N values
__device__ __forceinline__ i128 line_moment(const SpanStats& s, uint32_t N) {
  return 2 * s.T1 - mul_i128_u64(s.T0, N - 1);
}

// Sums of w and x w as high and low halves of w (the high half signed), each below 2^62 in magnitude
// while a thread adds at most 2^11 values at positions x < 2^17.
struct HalfSums {
  int64_t h0 = 0, l0 = 0, h1 = 0, l1 = 0;
  int64_t mn = INT64_MAX, mx = INT64_MIN;
  template <typename T>
  __device__ __forceinline__ void add(T value, uint32_t x) {
    const int64_t w = (int64_t)value;
    mn = min(mn, w);
    mx = max(mx, w);
    l0 += (int64_t)(uint32_t)w;
    l1 += (int64_t)((uint64_t)(uint32_t)w * x);
    if (sizeof(T) == 8) {
      h0 += (int64_t)(int32_t)(w >> 32);
      h1 += (int64_t)(int32_t)(w >> 32) * (int64_t)x;
    }
  }
  __device__ __forceinline__ SpanStats stats() const {
    SpanStats s;
    s.T0 = (i128)h0 * ((i128)1 << 32) + (i128)l0;
    s.T1 = (i128)h1 * ((i128)1 << 32) + (i128)l1;
    s.mn = mn;
    s.mx = mx;
    return s;
  }
};

// a span's moments from those of its differences from ref: Sd = sum d and its least-squares moment S
__device__ __forceinline__ SpanStats stats_from(int64_t ref, uint32_t N, int64_t Sd, int64_t S, int32_t mn, int32_t mx) {
  SpanStats s;
  s.T0 = mul_s64(ref, (int64_t)N) + (i128)Sd;
  s.T1 = ((i128)S + mul_i128_u64(s.T0, N - 1)) >> 1;  // S = 2 T1 - (N - 1) T0
  s.mn = ref + mn;
  s.mx = ref + mx;
  return s;
}

// moments of a short span by one thread
template <typename T>
__device__ __forceinline__ SpanStats lane_stats(const T* p, uint32_t N) {
  HalfSums h;
#pragma unroll 4
  for (uint32_t x = 0; x < N; x++) h.add(p[x], x);
  return h.stats();
}

// moments of the positions rank, rank + step, ... of a span of up to 2^16 values, summed over the tile
// (every lane has the sum)
template <int TILE, typename T>
__device__ __forceinline__ SpanStats group_stats(const T* p, uint32_t rank, uint32_t N, uint32_t step) {
  HalfSums h;
#pragma unroll 8
  for (uint32_t x = rank; x < N; x += step) h.add(p[x], x);
  h.l0 = tile_sum<TILE>(h.l0);
  h.l1 = tile_sum<TILE>(h.l1);
  if (sizeof(T) == 8) {
    h.h0 = tile_sum<TILE>(h.h0);
    h.h1 = tile_sum<TILE>(h.h1);
  }
  h.mn = tile_min<TILE>(h.mn);
  h.mx = tile_max<TILE>(h.mx);
  return h.stats();
}

// residual range at the positions x, x + step, ... < N under the parameters P (fit.cuh, steps 4
// and the fallback's widest zigzag residual), accumulated into lo, hi, zmax
template <typename T>
__device__ __forceinline__ void resid_part(const T* p, uint32_t x, uint32_t N, uint32_t step, const FitParams& P,
                                           int64_t& lo, int64_t& hi, uint64_t& zmax) {
  if (P.fallback) {
#pragma unroll 4
    for (; x < N; x += step) zmax = max(zmax, zz_encode((int64_t)((uint64_t)p[x] - (uint64_t)P.fb_shift)));
    return;
  }
  uint64_t F = (uint64_t)P.B * x;
  const uint64_t dF = (uint64_t)P.B * step;
  if (P.s >= 0) {
#pragma unroll 8
    for (; x < N; x += step, F += dF) {
      const int64_t r = (int64_t)p[x] - ((int64_t)F >> P.s);
      lo = min(lo, r);
      hi = max(hi, r);
    }
  } else {
#pragma unroll 4
    for (; x < N; x += step, F += dF) {
      const int64_t r = (int64_t)p[x] - (int64_t)(F << (-P.s));
      lo = min(lo, r);
      hi = max(hi, r);
    }
  }
}

}  // namespace
}  // namespace leco
