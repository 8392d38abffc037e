// Variable-length partitioning on the GPU (§3.2.2): split, then merge.
//
// Split: the sequence is cut into chunks of kChunk values (chunk edges always start a partition);
// inside a chunk partitions grow left to right: v_j joins the open partition [i, j) iff
// C = (j+1-i) D(v[i,j+1)) - (j-i) D(v[i,j)) <= tau * S_M and j - i < cap, where D is the linear
// regressor's fast metric bitlen(max d - min d) over the inner differences d_k = w_k - w_{k-1}. A CTA
// takes a chunk: its lanes sweep segments of it speculatively and one warp joins them to the sweep from
// the chunk's start (k_split). Starts go to a bitmap, which a count and a scan compact.
//
// Merge, round-synchronous: each round computes for every adjacent pair the size of the merged
// partition with the full regressor (S_M + len * b) and its gain over the two apart; every pair
// with a positive gain whose priority (gain, SplitMix64 of its start) beats both neighbouring
// pairs merges, all at once. Rounds repeat until none merges. Pair sizes are cached: only pairs
// touching a partition merged in the previous round are refitted, and a refit needs one pass over
// the pair's values, because every partition carries the moments of its values and two
// partitions' moments combine exactly (see SpanStats). The fits of the final partitions are the
// column's records, so the encoder does not fit them again.
#include <math.h>

#include <map>
#include <type_traits>
#include <vector>

#include "fit.cuh"
#include "leco_internal.cuh"
#include "span_fit.cuh"
#include "var_partition.cuh"

namespace leco {

cudaError_t scan_u64(const uint64_t* in, uint64_t count, uint64_t* out, uint64_t* scratch,
                     uint64_t* total, cudaStream_t st);

namespace {

constexpr uint64_t kChunk = 1ull << 16;

// ----------------------------------------------------------------------------------------- split
//
// A sweep opens a partition at its first value u_0 and grows it: with the open partition [i, j) of
// len = j - i values, metric cur = bitlen(max d - min d) over its differences, and next the metric
// with u_j's difference, u_j joins iff C = (len + 1) next - len cur <= floor(tau S_M) and len < cap
// (integers: for a real t, C <= t exactly when C <= floor(t)); a refused u_j opens the next partition.
//
// The chain of decisions is serial, but everything after a cut depends on the cut's position alone.
// So a CTA cuts the sweep into kSplitThreads segments and each lane runs two speculative sweeps over
// its own segment, one opened at the segment's first position and one at its second (two, because
// noisy columns cut every second value and a sweep then never leaves its parity). Once the true sweep
// cuts where a speculative one does, the two agree to the segment's end. Each lane then runs both
// sweeps 64 positions on into the next segment, to the first cut they share with that segment's
// speculative ones; one warp finally walks the segments: a table look-up where the true sweep was met
// (98 % of segments of the noisy columns, 65 - 80 % of the timestamps), else 32 candidates at a time
// until it is. All of it is exact; only the time depends on where sweeps meet.
// One lane or one warp per 65536-value chunk, as before, left the GPU to a chain of 65536 steps:
// 100M piecewise uint64 5.36 -> 0.54 ms, 250M 32-bit timestamps 1.81 -> 1.45 ms, a 30K column's whole
// partition + encode 2.9 -> 0.66 ms, 20M values split from seeds 37 -> 13 ms.
constexpr int kSplitThreads = 128;
constexpr uint32_t kSplitSegMax = (uint32_t)(kChunk / kSplitThreads);  // 512 positions
constexpr uint32_t kSplitWords = kSplitSegMax / 64;
constexpr uint32_t kNoCut = ~0u;

// the values u_k = v[base + dir k], k < count, of one sweep; vec: 32-byte loads of eight (dir = 1 and
// 32-byte aligned at every multiple of 8)
template <typename T>
struct SweepSrc {
  const T* __restrict__ v;
  uint64_t base;
  int dir;
  uint32_t count;
  bool vec;
  __device__ __forceinline__ T at(uint32_t k) const {
    return __ldg(v + (dir > 0 ? base + k : base - k));
  }
  // u_k .. u_{k+7} (k a multiple of 8); 0 past the end. A lane walks its own segment, so its loads
  // take whole sectors and ask L2 for the lines around them.
  __device__ __forceinline__ void at8(uint32_t k, T (&x)[8]) const {
    if (vec && k + 8 <= count) {
      const T* p = v + base + k;
      if (sizeof(T) == 8) {
        unsigned long long t[8];
        asm("ld.global.nc.L2::256B.v4.u64 {%0,%1,%2,%3}, [%4];"
            : "=l"(t[0]), "=l"(t[1]), "=l"(t[2]), "=l"(t[3])
            : "l"(p));
        asm("ld.global.nc.L2::256B.v4.u64 {%0,%1,%2,%3}, [%4];"
            : "=l"(t[4]), "=l"(t[5]), "=l"(t[6]), "=l"(t[7])
            : "l"(p + 4));
#pragma unroll
        for (int u = 0; u < 8; u++) x[u] = (T)t[u];
      } else {
        uint32_t t[8];
        asm("ld.global.nc.L2::256B.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]), "=r"(t[7])
            : "l"(p));
#pragma unroll
        for (int u = 0; u < 8; u++) x[u] = (T)t[u];
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; u++) x[u] = k + u < count ? at(k + u) : (T)0;
    }
  }
};

// differences and their extremes: int64 for values in (-2^62, 2^62) as int64 (the range of two
// differences then stays below 2^64, taken unsigned), else 128-bit
template <typename D>
__device__ __forceinline__ D d_lowest();
template <>
__device__ __forceinline__ int64_t d_lowest<int64_t>() {
  return INT64_MIN;
}
template <>
__device__ __forceinline__ i128 d_lowest<i128>() {
  return -((i128)1 << 100);
}
template <typename D>
__device__ __forceinline__ D d_highest();
template <>
__device__ __forceinline__ int64_t d_highest<int64_t>() {
  return INT64_MAX;
}
template <>
__device__ __forceinline__ i128 d_highest<i128>() {
  return (i128)1 << 100;
}
__device__ __forceinline__ int d_metric(int64_t mx, int64_t mn) { return bitlen_u64((uint64_t)mx - (uint64_t)mn); }
__device__ __forceinline__ int d_metric(i128 mx, i128 mn) { return bitlen_u128((u128)(mx - mn)); }
__device__ __forceinline__ int64_t d_shfl_up(int64_t v, uint32_t o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ i128 d_shfl_up(i128 v, uint32_t o) {
  const uint64_t lo = __shfl_up_sync(0xffffffffu, (uint64_t)v, o);
  const uint64_t hi = __shfl_up_sync(0xffffffffu, (uint64_t)((u128)v >> 64), o);
  return (i128)(((u128)hi << 64) | lo);
}
__device__ __forceinline__ int64_t d_shfl(int64_t v, uint32_t src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ i128 d_shfl(i128 v, uint32_t src) {
  const uint64_t lo = __shfl_sync(0xffffffffu, (uint64_t)v, src);
  const uint64_t hi = __shfl_sync(0xffffffffu, (uint64_t)((u128)v >> 64), src);
  return (i128)(((u128)hi << 64) | lo);
}

// an open partition: the extremes of its differences, its metric and its length. len = cap makes the
// next step cut whatever its value is.
template <typename D>
struct Sweep {
  D mx, mn;
  int cur;
  uint32_t len;
  // the next value, at difference d from its predecessor: true when it is refused and opens a partition
  __device__ __forceinline__ bool step(D d, uint32_t cap, int tf) {
    const D a = d > mx ? d : mx, b = d < mn ? d : mn;
    const int next = d_metric(a, b);
    const int C = (int)len * (next - cur) + next;  // (len + 1) next - len cur; len <= 2^16, metrics <= 66
    const bool cut = C > tf || len >= cap;
    mx = cut ? d_lowest<D>() : a;
    mn = cut ? d_highest<D>() : b;
    cur = cut ? 0 : next;
    len = cut ? 1u : len + 1u;
    return cut;
  }
};

struct SplitShared {
  uint64_t bits[2][kSplitThreads * kSplitWords];  // cuts of the two speculative sweeps; [0] becomes the result
  uint64_t over[2][kSplitThreads];                // their cuts in the 64 positions after the segment
  int64_t ext[2][kSplitThreads];                  // extremes of the first sweep's last partition
  uint16_t last[kSplitThreads];                   // its start, relative to the segment (kNoLast: not known)
  uint8_t met[2][kSplitThreads];                  // position and sweep of the first shared cut, kMet when there is one
};
constexpr uint8_t kMet = 0x80, kMetSecond = 0x40;
constexpr uint16_t kNoLast = 0xFFFF;

// both speculative sweeps over the lane's segment [s, t), nw words of 64 positions; returns whether a
// value lies outside (-2^62, 2^62)
template <typename D, typename T>
__device__ __forceinline__ bool lane_segment(const SweepSrc<T>& src, uint32_t s, uint32_t t, uint32_t cap, int tf,
                                             uint64_t* bitsA, uint64_t* bitsB, Sweep<D>& A, Sweep<D>& B, T& prev) {
  const int64_t lim = (int64_t)1 << 62;
  bool wide = false;
  A.mx = B.mx = d_lowest<D>();
  A.mn = B.mn = d_highest<D>();
  A.cur = B.cur = 0;
  A.len = B.len = cap;
  prev = s && s < t ? src.at(s - 1) : (T)0;
  T nx[8];
  if (s < t) src.at8(s, nx);
  for (uint32_t k = s; k < t; k += 64) {
    uint64_t wa = 0, wb = 0;
    for (uint32_t y = 0; y < 64 && k + y < t; y += 8) {
      T x[8];
#pragma unroll
      for (int u = 0; u < 8; u++) x[u] = nx[u];
      if (k + y + 8 < t) src.at8(k + y + 8, nx);
      uint32_t ca = 0, cb = 0;
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const int64_t w = (int64_t)x[u];
        if (sizeof(T) == 8) wide = wide || w <= -lim || w >= lim;
        const D d = (D)w - (D)(int64_t)prev;
        prev = x[u];
        ca |= A.step(d, cap, tf) ? 1u << u : 0u;
        cb |= B.step(d, cap, tf) ? 1u << u : 0u;
        if (u == 0 && k + y == s) B.len = cap;  // the second sweep opens at the second position
      }
      wa |= (uint64_t)ca << y;
      wb |= (uint64_t)cb << y;
    }
    const uint64_t keep = t - k >= 64 ? ~0ull : (1ull << (t - k)) - 1ull;
    bitsA[(k - s) >> 6] = wa & keep;
    bitsB[(k - s) >> 6] = wb & keep & (k == s ? ~1ull : ~0ull);
  }
  return wide;
}

// both sweeps 64 positions on from t, and the first cut each shares with the next segment's sweeps
template <typename D, typename T>
__device__ __forceinline__ void lane_overrun(const SweepSrc<T>& src, uint32_t t, uint32_t cap, int tf, Sweep<D>& A,
                                             Sweep<D>& B, T prev, SplitShared& sh, uint32_t seg, uint32_t nw) {
  uint64_t oa = 0, ob = 0;
  for (uint32_t y = 0; y < 64; y += 8) {
    T x[8];
    src.at8(t + y, x);
    uint32_t ca = 0, cb = 0;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const D d = (D)(int64_t)x[u] - (D)(int64_t)prev;
      prev = x[u];
      ca |= A.step(d, cap, tf) ? 1u << u : 0u;
      cb |= B.step(d, cap, tf) ? 1u << u : 0u;
    }
    oa |= (uint64_t)ca << y;
    ob |= (uint64_t)cb << y;
  }
  const uint64_t na = sh.bits[0][(seg + 1) * nw], nb = sh.bits[1][(seg + 1) * nw];
  auto meet = [&](uint64_t o) -> uint8_t {
    const uint64_t h = o & (na | nb);
    if (!h) return 0;
    const int x = __ffsll((long long)h) - 1;
    return (uint8_t)(kMet | ((na >> x) & 1ull ? 0u : kMetSecond) | (uint32_t)x);
  };
  sh.over[0][seg] = oa;
  sh.over[1][seg] = ob;
  sh.met[0][seg] = meet(oa);
  sh.met[1][seg] = meet(ob);
}

// The true sweep over the segments by one warp, from the speculative ones: bits[0] becomes its cuts.
template <typename D, typename T>
__device__ void walk_segments(const SweepSrc<T>& src, uint32_t seglen, uint32_t nseg, uint32_t cap, int tf,
                              SplitShared& sh) {
  const uint32_t lane = threadIdx.x & 31u, nw = seglen >> 6;
  uint32_t which = 0;    // the speculative sweep of the segment before that the true sweep follows at its end
  bool live = false;     // ... or none: the open partition [i, j0) below
  uint32_t i = 0, j0 = 1;
  D cmax = d_lowest<D>(), cmin = d_highest<D>();
  int ccur = 0;
  // Candidates j0 .. lim - 1, 32 at a time: lane l assumes that every candidate before it joined, so
  // its extremes are the carried ones with an inclusive scan's, and the metric before it is the lane
  // below's. Stops at the first refusal (returned; the partition it opens is then the open one) or at
  // j0 = lim. A window that leaves the metric unchanged joins whole: every C in it is the metric.
  auto advance = [&](uint32_t lim) -> uint32_t {
    T nx = j0 + lane < lim ? src.at(j0 + lane) : (T)0;
    T before = j0 < lim ? src.at(j0 - 1) : (T)0;
    while (j0 < lim) {
      const T w = nx;
      const uint32_t j = j0 + lane;
      const bool valid = j < lim;
      nx = j + 32 < lim ? src.at(j + 32) : (T)0;
      T pw = __shfl_up_sync(0xffffffffu, w, 1);
      if (lane == 0) pw = before;
      const D d = valid ? (D)(int64_t)w - (D)(int64_t)pw : (D)0;
      const uint32_t last = lim - j0 < 32u ? lim - j0 - 1 : 31u;
      if (sizeof(D) == 8 && __all_sync(0xffffffffu, d >= (D)INT32_MIN && d <= (D)INT32_MAX)) {
        const int32_t wmax = __reduce_max_sync(0xffffffffu, valid ? (int32_t)d : INT32_MIN);
        const int32_t wmin = __reduce_min_sync(0xffffffffu, valid ? (int32_t)d : INT32_MAX);
        const D amax = cmax > (D)wmax ? cmax : (D)wmax, amin = cmin < (D)wmin ? cmin : (D)wmin;
        if (d_metric(amax, amin) == ccur && ccur <= tf && j0 + last - i < cap) {
          cmax = amax;
          cmin = amin;
          before = __shfl_sync(0xffffffffu, w, last);
          j0 += last + 1;
          continue;
        }
      }
      D pmax = valid ? d : d_lowest<D>(), pmin = valid ? d : d_highest<D>();
#pragma unroll
      for (uint32_t o = 1; o < 32; o <<= 1) {
        const D tmax = d_shfl_up(pmax, o), tmin = d_shfl_up(pmin, o);
        if (lane >= o) {
          pmax = tmax > pmax ? tmax : pmax;
          pmin = tmin < pmin ? tmin : pmin;
        }
      }
      const D nmax = cmax > pmax ? cmax : pmax, nmin = cmin < pmin ? cmin : pmin;
      const int next = d_metric(nmax, nmin);
      int cur = __shfl_up_sync(0xffffffffu, next, 1);
      if (lane == 0) cur = ccur;
      const uint32_t len = j - i;
      const int C = (int)len * (next - cur) + next;
      const uint32_t rej = __ballot_sync(0xffffffffu, valid && (C > tf || len >= cap));
      if (rej) {
        const uint32_t at = j0 + (uint32_t)(__ffs(rej) - 1);
        cmax = d_lowest<D>();
        cmin = d_highest<D>();
        ccur = 0;
        i = at;
        j0 = at + 1;
        return at;
      }
      cmax = d_shfl(nmax, last);
      cmin = d_shfl(nmin, last);
      ccur = __shfl_sync(0xffffffffu, next, last);
      before = __shfl_sync(0xffffffffu, w, last);
      j0 += last + 1;
    }
    return kNoCut;
  };
  for (uint32_t seg = 1; seg < nseg; seg++) {
    uint64_t* fin = sh.bits[0] + seg * nw;
    const uint64_t* second = sh.bits[1] + seg * nw;
    const uint32_t s = seg * seglen, t = min(s + seglen, src.count);
    if (!live) {
      const uint8_t m = sh.met[which][seg - 1];
      if (m & kMet) {
        const uint32_t x = m & 63u, w2 = (m & kMetSecond) ? 1u : 0u;
        const uint64_t below = (1ull << x) - 1ull, o = sh.over[which][seg - 1];
        if (lane < nw) {
          uint64_t w = w2 ? second[lane] : fin[lane];
          if (lane == 0) w = (w & ~below) | (o & below);
          fin[lane] = w;
        }
        which = w2;
        continue;
      }
      // not met in 64 positions: take the open partition from the last cut before the segment
      __syncwarp();
      const uint64_t w = lane < nw ? sh.bits[0][(seg - 1) * nw + lane] : 0;
      const uint32_t nz = __ballot_sync(0xffffffffu, w != 0);
      const int src_lane = 31 - __clz((int)nz);  // the segment holds a cut: the true sweep was met there
      const uint64_t lw = __shfl_sync(0xffffffffu, w, src_lane);
      i = (seg - 1) * seglen + (uint32_t)src_lane * 64u + (uint32_t)(63 - __clzll((long long)lw));
      j0 = i + 1;
      cmax = d_lowest<D>();
      cmin = d_highest<D>();
      ccur = 0;
      advance(s);  // no cut lies between
      live = true;
    }
    uint64_t cuts = 0;  // lane w < nw: the true cuts found so far in word w
    const uint32_t lastA = s + sh.last[seg];
    bool tail = sizeof(D) == 8 && sh.last[seg] != kNoLast;  // the first sweep's last partition may join whole
    for (;;) {
      if (tail && j0 == lastA + 1) {
        const D emax = (D)sh.ext[0][seg], emin = (D)sh.ext[1][seg];
        const D amax = cmax > emax ? cmax : emax, amin = cmin < emin ? cmin : emin;
        tail = false;
        if (j0 < t && d_metric(amax, amin) == ccur && ccur <= tf && t - 1 - i < cap) {
          cmax = amax;
          cmin = amin;
          j0 = t;
        }
      }
      if (j0 >= t) break;
      const uint32_t at = advance(tail && j0 <= lastA ? lastA + 1 : t);
      if (at == kNoCut) continue;
      const uint32_t r = at - s;
      const bool inA = (fin[r >> 6] >> (r & 63u)) & 1ull, inB = (second[r >> 6] >> (r & 63u)) & 1ull;
      if (inA || inB) {
        __syncwarp();
        if (lane < nw) {
          const uint64_t from = lane < (r >> 6) ? 0ull : (lane == (r >> 6) ? ~0ull << (r & 63u) : ~0ull);
          fin[lane] = cuts | ((inA ? fin[lane] : second[lane]) & from);
        }
        which = inA ? 0u : 1u;
        live = false;
        break;
      }
      if (lane == (r >> 6)) cuts |= 1ull << (r & 63u);
    }
    if (live) {
      __syncwarp();
      if (lane < nw) fin[lane] = cuts;
    }
    __syncwarp();
  }
}

// One sweep per CTA. SEEDED = false: chunk c forwards from its first value. SEEDED (§3.2.2, selecting
// good starting positions): CTA 2c sweeps chunk c forwards from its seed, CTA 2c + 1 backwards from the
// value before the seed with the same rule (a partition refused there at u_k starts at seed - k); the
// chunk edge and the seed are cuts, and the bitmap, shared by both, is zero on entry.
template <typename T, bool SEEDED>
__global__ void __launch_bounds__(kSplitThreads)
    k_split(const T* __restrict__ v, uint64_t n, uint32_t cap_in, int64_t tfloor, const uint64_t* __restrict__ seeds,
            uint64_t* __restrict__ bitmap) {
  __shared__ SplitShared sh;
  const uint64_t c = SEEDED ? blockIdx.x >> 1 : blockIdx.x;
  const uint64_t a = c * kChunk, e = min(a + kChunk, n);
  const uint64_t seed = SEEDED ? seeds[c] : a;
  const bool back = SEEDED && (blockIdx.x & 1u);
  SweepSrc<T> src;
  src.v = v;
  src.base = back ? seed - 1 : seed;
  src.dir = back ? -1 : 1;
  src.count = (uint32_t)(back ? seed - a : e - seed);
  src.vec = !SEEDED && (reinterpret_cast<uintptr_t>(v) & 31u) == 0;
  if (src.count == 0) return;  // backwards from a seed at the chunk's edge
  const uint32_t cap = cap_in < 2u * (uint32_t)kChunk ? cap_in : 2u * (uint32_t)kChunk;
  const int tf = tfloor > (int64_t)INT32_MAX ? INT32_MAX : (int)tfloor;
  const uint32_t seglen = ((src.count + kSplitThreads - 1) / kSplitThreads + 63u) & ~63u;  // 64 .. 512
  const uint32_t nseg = (src.count + seglen - 1) / seglen, nw = seglen >> 6;
  const uint32_t seg = threadIdx.x;
  const uint32_t s = min(seg * seglen, src.count), t = min(s + seglen, src.count);
  uint64_t *ba = sh.bits[0] + seg * nw, *bb = sh.bits[1] + seg * nw;
  T prev;
  Sweep<int64_t> A, B;
  bool wide = lane_segment(src, s, t, cap, tf, ba, bb, A, B, prev);
  wide = __syncthreads_or(wide);
  if (!wide) {
    if (seg < nseg) {
      sh.ext[0][seg] = A.mx;
      sh.ext[1][seg] = A.mn;
      // (a lane's steps go on to a multiple of eight: past the end in the last segment)
      sh.last[seg] = (t - s) & 7u ? kNoLast : (uint16_t)(t - s - A.len);
    }
    if (seg + 1 < nseg) lane_overrun(src, t, cap, tf, A, B, prev, sh, seg, nw);
    __syncthreads();
    if (seg < 32) walk_segments<int64_t>(src, seglen, nseg, cap, tf, sh);
  } else {
    Sweep<i128> A2, B2;
    lane_segment(src, s, t, cap, tf, ba, bb, A2, B2, prev);
    __syncthreads();
    if (seg + 1 < nseg) lane_overrun(src, t, cap, tf, A2, B2, prev, sh, seg, nw);
    __syncthreads();
    if (seg < 32) walk_segments<i128>(src, seglen, nseg, cap, tf, sh);
  }
  __syncthreads();
  const uint32_t words = (src.count + 63) >> 6;
  const uint64_t* fin = sh.bits[0];
  if (!SEEDED) {
    for (uint32_t w = threadIdx.x; w < words; w += kSplitThreads) bitmap[(a >> 6) + w] = fin[w];
    return;
  }
  const uint64_t first = back ? a : seed, g0 = first >> 6, g1 = (back ? seed : e - 1) >> 6;
  for (uint64_t g = g0 + threadIdx.x; g <= g1; g += kSplitThreads) {
    // bit b of the word is position 64 g + b: u-index 64 g + b - seed forwards, seed - 64 g - b backwards
    const int64_t k = back ? (int64_t)seed - (int64_t)(64 * g) - 63 : (int64_t)(64 * g) - (int64_t)seed;
    const uint32_t q = k >= 0 ? (uint32_t)k >> 6 : 0u, o = (uint32_t)k & 63u;  // k > -64
    uint64_t x;
    if (k < 0)
      x = fin[0] << (uint32_t)(-k);
    else
      x = (q < words ? fin[q] >> o : 0ull) | (o && q + 1 < words ? fin[q + 1] << (64u - o) : 0ull);
    if (back) x = __brevll(x);
    if (x) atomicOr((unsigned long long*)&bitmap[g], (unsigned long long)x);
  }
  if (threadIdx.x == 0) atomicOr((unsigned long long*)&bitmap[a >> 6], 1ull << (a & 63u));
}

// seed[c] = the first k of chunk c whose second-order delta w_{k+2} - 2 w_{k+1} + w_k has the
// shortest zigzag code (the linear regressor's smoothest window); the chunk's first position when
// it holds fewer than 3 values. A CTA per chunk; the (bits, k) minimum is reduced over the CTA.
template <typename T>
__global__ void __launch_bounds__(256) k_chunk_seed(const T* __restrict__ v, uint64_t n, uint64_t* __restrict__ seed) {
  __shared__ uint64_t red[8];
  const uint64_t nchunks = (n + kChunk - 1) / kChunk;
  for (uint64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const uint64_t a = c * kChunk, e = min(a + kChunk, n);
    uint64_t best = ~0ull;  // bits << 32 | (k - a): the minimum is the smallest bits, then the first k
    for (uint64_t k = a + threadIdx.x; k + 2 < e; k += blockDim.x) {
      const i128 d2 = (i128)(int64_t)__ldg(v + k + 2) - 2 * (i128)(int64_t)__ldg(v + k + 1) + (i128)(int64_t)__ldg(v + k);
      const u128 z = d2 >= 0 ? (u128)d2 * 2 : (u128)(-d2) * 2 - 1;
      const uint64_t key = ((uint64_t)bitlen_u128(z) << 32) | (k - a);
      best = key < best ? key : best;
    }
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t t = __shfl_down_sync(0xffffffffu, best, o);
      best = t < best ? t : best;
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = best;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; w++) best = red[w] < best ? red[w] : best;
      seed[c] = best == ~0ull ? a : a + (best & 0xFFFFFFFFull);
    }
    __syncthreads();
  }
}

// starts per chunk (a CTA per chunk, 1024 bitmap words)
__global__ void __launch_bounds__(256) k_count_starts(const uint64_t* __restrict__ bitmap, uint64_t nw,
                                                      uint64_t* __restrict__ cnt) {
  __shared__ uint32_t ws[8];
  const uint64_t w0 = blockIdx.x * (kChunk / 64);
  uint32_t k = 0;
  for (uint64_t w = w0 + threadIdx.x; w < min(w0 + kChunk / 64, nw); w += 256) k += (uint32_t)__popcll(bitmap[w]);
  k = __reduce_add_sync(0xffffffffu, k);
  if ((threadIdx.x & 31u) == 0) ws[threadIdx.x >> 5] = k;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int j = 1; j < 8; j++) k += ws[j];
    cnt[blockIdx.x] = k;
  }
}

// The starts of one chunk (a CTA): the words' ranks by a scan over the CTA, then a warp spreads each
// word, lane l the bits l and l + 32, so that the stores of one word lie side by side (a thread per
// word, as before, took 495 us for the 44M starts of 100M piecewise values; this way 68 us).
__global__ void __launch_bounds__(256) k_scatter_starts(const uint64_t* __restrict__ bitmap, uint64_t nw,
                                                        const uint64_t* __restrict__ pos, uint64_t n, uint64_t m,
                                                        uint64_t* __restrict__ starts) {
  __shared__ uint64_t words[kChunk / 64];
  __shared__ uint32_t rank[kChunk / 64];
  __shared__ uint32_t ws[8];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const uint64_t w0 = blockIdx.x * (kChunk / 64);
  const uint32_t words_here = (uint32_t)(min(w0 + kChunk / 64, nw) - w0);
  uint32_t c[4], sum = 0;
  for (int u = 0; u < 4; u++) {
    const uint32_t w = t * 4 + u;
    const uint64_t x = w < words_here ? bitmap[w0 + w] : 0;
    words[w] = x;
    c[u] = (uint32_t)__popcll(x);
    sum += c[u];
  }
  uint32_t inc = sum;
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  uint32_t r = inc - sum;
  for (uint32_t w = 0; w < warp; w++) r += ws[w];
  for (int u = 0; u < 4; u++) {
    rank[t * 4 + u] = r;
    r += c[u];
  }
  __syncthreads();
  uint64_t* out = starts + pos[blockIdx.x];
  const uint64_t base = w0 * 64;
  for (uint32_t w = warp; w < words_here; w += 8) {
    const uint64_t x = words[w];
    const uint32_t lo = (uint32_t)x, hi = (uint32_t)(x >> 32), below = (1u << lane) - 1u, q = rank[w];
    if ((lo >> lane) & 1u) out[q + __popc(lo & below)] = base + w * 64ull + lane;
    if ((hi >> lane) & 1u) out[q + __popc(lo) + __popc(hi & below)] = base + w * 64ull + 32 + lane;
  }
  if (blockIdx.x == 0 && t == 0) starts[m] = n;
}

// Fixed-partition size search (§3.2.1): total S_M + len * b over partitions of L values cut from
// each of k sampled subsequences of N values (starts[s]), the last of each possibly short.
// Thread per partition for L <= kTinySpan, warp per partition above; one atomic per warp.
__global__ void k_sample_sizes_thread(const void* __restrict__ values, int dtype, const uint64_t* __restrict__ starts,
                                      uint64_t k, uint32_t N, uint32_t L, int model,
                                      unsigned long long* __restrict__ total) {
  const uint64_t P = (N + L - 1) / L, count = k * P;
  uint64_t acc = 0;
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < count; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t s = t / P, j = t - s * P;
    const uint32_t len = (uint32_t)min((uint64_t)L, (uint64_t)N - j * L);
    const FitResult R = fit_range<1>(values, dtype, starts[s] + j * L, len, model, 0, nullptr);
    acc += kSmBits + (uint64_t)len * R.b;
  }
  acc = warp_sum_u64(acc);
  if ((threadIdx.x & 31u) == 0 && acc) atomicAdd(total, (unsigned long long)acc);
}

__global__ void k_sample_sizes_warp(const void* __restrict__ values, int dtype, const uint64_t* __restrict__ starts,
                                    uint64_t k, uint32_t N, uint32_t L, int model,
                                    unsigned long long* __restrict__ total) {
  const uint64_t P = (N + L - 1) / L, count = k * P;
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  uint64_t acc = 0;
  for (uint64_t t = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; t < count; t += nw) {
    const uint64_t s = t / P, j = t - s * P;
    const uint32_t len = (uint32_t)min((uint64_t)L, (uint64_t)N - j * L);
    const FitResult R = fit_range<32>(values, dtype, starts[s] + j * L, len, model, lane, nullptr);
    acc += kSmBits + (uint64_t)len * R.b;
  }
  if (lane == 0 && acc) atomicAdd(total, (unsigned long long)acc);
}

int grid_for(uint64_t items, int per_block, int max_blocks_per_sm) {
  const uint64_t need = (items + per_block - 1) / per_block;
  const uint64_t cap = (uint64_t)sm_count() * max_blocks_per_sm;
  return (int)(need < cap ? (need ? need : 1) : cap);
}

// ----------------------------------------------------------------------------------------- merge
//
// A partition is its start, its width b (a byte; its size is S_M + len b) and, beyond kStatVals values,
// its values' moments (SpanStats, span_fit.cuh). The moments sit in a table by start / 32, where partitions
// of more than 32 values never collide: they stay in place when partitions merge, so a round moves ten
// bytes per partition. Shorter partitions' moments are taken from their values whenever they are needed,
// which reads less than storing them would. A pair is its left partition's merged width mb, or
//   kDirty  not fitted since one of its partitions changed,
//   kNo     no gain (a pair that does not gain never merges and never keeps a neighbour from merging: its
//           width does not matter) or longer than the cap.
// While most pairs change (dense rounds) a round is: k_fit_spans (a lane fits a pair of up to kLaneVals
// values by itself, from values the warp staged; longer pairs get their line there, from combined moments),
// k_span_range (a warp takes a longer pair's residual range and stops as soon as the range rules out a
// gain), k_select, a scan of the tiles' counts, k_merge_stats (moments of the merged), k_compact. Once few
// pairs merge (sparse rounds), partitions stay in their slots, linked left and right, and a round touches
// only the pairs that can merge and those that changed.
// Measured, 100M piecewise uint64 (45 rounds) and 250M 32-bit timestamps (62 rounds), against 16-byte sizes
// and 48-byte moments moved every round, one kernel of 78 registers for fits of all lengths, and ten
// launches and a host round trip per round to the end: whole passes 28.05 -> 20.46 ms and 18.37 -> 11.59 ms
// (17.7 and 10.3 ms with what the kernels below say of themselves).
constexpr uint32_t kTinySpan = 256;    // size search: a thread per sampled partition up to this size
constexpr uint32_t kLaneVals = 64;     // a lane fits spans up to this long on its own
constexpr uint32_t kStatVals = 32;     // longer partitions carry their moments (at most kLaneVals; the table's stride)
constexpr uint32_t kPieceVals = 4096;  // a warp takes the residual range of a span up to this long; pieces above
constexpr int kSpanBlock = 128;        // k_fit_spans: 4 warps, each taking 32 spans at a time
constexpr uint32_t kSpanStage = 1088;  // staged differences per warp
constexpr uint32_t kTileVals = 512;    // spans up to this long take eight lanes, four at a time, longer ones a warp
constexpr uint8_t kNo = 0xFF, kDirty = 0xFE, kDead = 0xFD;
constexpr uint32_t kSlotEnd = 0xFFFFFFFFu;
// sparse rounds begin below one merge in kSparseShare partitions, or at kSparseBelow partitions, where a dense
// round's launches and host round trip cost more than its work
constexpr uint64_t kSparseShare = 16, kSparseBelow = 32768;

// a longer span and its line (fallback: B is the shift); bmax: widths above it bring no gain
struct SpanJob {
  uint64_t a;
  int64_t B;
  uint64_t j;
  uint32_t N;
  int8_t s;
  uint8_t fallback;
  uint8_t bmax;
  uint8_t narrow;  // values within 2^30 of each other, line within 2^30 (span_fit.cuh)
};
static_assert(sizeof(SpanJob) == 32, "span job layout");

// piece q of np of a job beyond kPieceVals, whose range is gathered in slot mi
struct SpanPiece {
  uint32_t e, mi, q, np;
};

struct SpanWork {
  SpanJob* jobs;
  SpanPiece* pieces;
  long long *lo, *hi;  // per slot
  unsigned long long* zmax;
  uint32_t* done;
  unsigned long long* cnt;  // jobs, pieces, slots
};

// a span's job (and pieces) at place e of the list
__device__ __forceinline__ void put_job(const SpanWork& w, uint64_t e, uint64_t a, uint32_t N, uint64_t j,
                                        const FitParams& P, uint32_t bmax, bool narrow, bool pieces) {
  SpanJob q;
  q.a = a;
  q.B = P.fallback ? P.fb_shift : P.B;
  q.j = j;
  q.N = N;
  q.s = (int8_t)P.s;
  q.fallback = (uint8_t)P.fallback;
  q.bmax = (uint8_t)bmax;
  q.narrow = narrow ? 1 : 0;
  w.jobs[e] = q;
  if (!pieces || N <= kPieceVals) return;
  const uint32_t np = (N + kPieceVals - 1) / kPieceVals;
  const unsigned long long mi = atomicAdd(&w.cnt[2], 1ull), pb = atomicAdd(&w.cnt[1], (unsigned long long)np);
  w.lo[mi] = INT64_MAX;
  w.hi[mi] = INT64_MIN;
  w.zmax[mi] = 0;
  w.done[mi] = 0;
  for (uint32_t k = 0; k < np; k++) w.pieces[pb + k] = SpanPiece{(uint32_t)e, (uint32_t)mi, k, np};
}

// the largest width that gains when partitions of N1 and N2 values and widths b1 and b2 merge:
// S_M + N b < 2 S_M + N1 b1 + N2 b2
__device__ __forceinline__ uint32_t gain_width(uint32_t N1, uint32_t b1, uint32_t N2, uint32_t b2) {
  return min(((uint32_t)kSmBits + N1 * b1 + N2 * b2 - 1u) / (N1 + N2), 64u);  // lengths below 2^25, widths up to 64
}

__device__ __forceinline__ Record span_record(uint64_t a, const FitResult& R) {
  Record r;
  r.theta0 = R.theta0;
  r.theta1 = R.theta1;
  r.start = a;
  r.word3 = make_w3(0, R.b, R.s, 1);
  return r;
}

// the moments of a partition: from the table, or from its values when it is short
template <typename T>
__device__ __forceinline__ SpanStats part_stats(const T* __restrict__ v, uint64_t a, uint32_t N,
                                                const SpanStats* __restrict__ stats) {
  return N > kStatVals ? stats[a / kStatVals] : lane_stats(v + a, N);
}

template <typename T>
struct SpanArgs {
  const T* v;
  uint32_t cap;
  int model;
  SpanStats* stats;
  SpanWork w;
};

// Fits of the spans [st[j], st[j + W]), j < count, a lane each. MODE 1: the split's partitions (b[j];
// moments of those beyond kStatVals into the table; those beyond kLaneVals are listed for k_fit_long).
// MODE 2: the dirty pairs (W = 2; mb[j]). MODE 3: the final partitions (rec[j]). Spans beyond kLaneVals get
// their line from their moments and go to the job list. The warp stages the values of its short spans as
// 32-bit differences from the first one, which leaves both passes over them in 32 bits; values too far
// apart are read from memory in 64 bits instead.
template <typename T, int MODE>
__global__ void __launch_bounds__(kSpanBlock, 8)
    k_fit_spans(const SpanArgs<T> A, const uint64_t* __restrict__ st, uint64_t count, uint8_t* __restrict__ b,
                uint8_t* __restrict__ mb, Record* __restrict__ rec) {
  constexpr int W = MODE == 2 ? 2 : 1;
  __shared__ int32_t raw[kSpanBlock / 32][kSpanStage];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  int32_t* stage = raw[wib];
  const uint64_t groups = (count + 31) / 32, gw = (uint64_t)gridDim.x * (kSpanBlock / 32);
  for (uint64_t g = (uint64_t)blockIdx.x * (kSpanBlock / 32) + wib; g < groups; g += gw) {
    const uint64_t j = g * 32 + lane;
    bool act = j < count && (MODE != 2 || mb[j] == kDirty);
    if (!__any_sync(kFull, act)) continue;
    uint64_t a = 0, mid = 0, c = 0;
    uint32_t bmax = 64;
    if (act) {
      a = st[j];
      c = st[j + W];
      if (W == 2) {
        mid = st[j + 1];
        if (c - a > A.cap) {
          mb[j] = kNo;
          act = false;
        } else {
          bmax = gain_width((uint32_t)(mid - a), b[j], (uint32_t)(c - mid), b[j + 1]);
        }
      }
    }
    const uint32_t N = act ? (uint32_t)(c - a) : 0u;
    const bool small = act && N <= kLaneVals;
    const uint32_t smalls = __ballot_sync(kFull, small);
    uint64_t ga = 0;
    int64_t ref = 0;
    bool narrow = false;
    if (smalls) {  // their values, from the first one's start to the last one's end
      ga = __shfl_sync(kFull, a, __ffs((int)smalls) - 1);
      const uint64_t gc = __shfl_sync(kFull, c, 31 - __clz((int)smalls));
      if (gc - ga <= kSpanStage) {
        const uint32_t len = (uint32_t)(gc - ga);
        ref = (int64_t)__ldg(A.v + ga);
        bool ok = narrow_ref(ref);
#pragma unroll 4
        for (uint32_t t = lane; t < len; t += 32) {
          const int64_t d = (int64_t)__ldg(A.v + ga + t) - ref;
          ok = ok && narrow_diff(d);
          stage[t] = (int32_t)d;
        }
        narrow = __all_sync(kFull, ok);
        __syncwarp();
      }
    }
    const bool lin = A.model == LECO_MODEL_LINEAR && N >= 2;
    const int32_t* dp = stage + (uint32_t)(a - ga);
    SpanStats S;
    i128 moment = 0;
    S.T0 = S.T1 = 0;
    S.mn = S.mx = 0;
    if (small && narrow) {
      int64_t sum = 0, Sd = 0;
      int32_t mn = INT32_MAX, mx = INT32_MIN, u = 1 - (int32_t)N;  // u = 2 x - (N - 1)
#pragma unroll 4
      for (uint32_t x = 0; x < N; x++, u += 2) {
        const int32_t d = dp[x];
        mn = min(mn, d);
        mx = max(mx, d);
        sum += (int64_t)u * d;
        if (W == 1) Sd += d;
      }
      S.mn = ref + mn;
      S.mx = ref + mx;
      moment = sum;
      if (MODE == 1 && N > kStatVals) A.stats[a / kStatVals] = stats_from(ref, N, Sd, sum, mn, mx);
    } else if (small) {
      S = lane_stats(A.v + a, N);
      moment = line_moment(S, N);
      if (MODE == 1 && N > kStatVals) A.stats[a / kStatVals] = S;
    } else if (act && MODE != 1) {
      if (W == 2)
        S = combine_stats(part_stats(A.v, a, (uint32_t)(mid - a), A.stats), mid - a,
                          part_stats(A.v, mid, (uint32_t)(c - mid), A.stats));
      else
        S = A.stats[a / kStatVals];
      moment = line_moment(S, N);
    }
    FitParams P;
    P.B = 0;
    P.fb_shift = 0;
    P.s = 0;
    P.fallback = 0;
    if (act && (small || MODE != 1)) P = solve_params(lin ? moment : (i128)0, S.mx, S.mn, N, lin);
    // the residual range; the constant model's residuals on its grid are the values themselves
    int64_t lo = S.mn, hi = S.mx;
    uint64_t zmax = 0;
    const bool need = lin || P.fallback;
    const bool flat = act && narrow_line(P, N);
    if (small && need) {
      lo = INT64_MAX;
      hi = INT64_MIN;
      if (narrow && flat) {
        const NarrowLine line(P.B, P.s);
        int32_t l = INT32_MAX, h = INT32_MIN;
        uint64_t G = 0;
#pragma unroll 4
        for (uint32_t x = 0; x < N; x++, G += line.B) {
          const int32_t r = dp[x] - line.at(G);
          l = min(l, r);
          h = max(h, r);
        }
        lo = ref + l;
        hi = ref + h;
      } else {
        resid_part(A.v + a, 0, N, 1, P, lo, hi, zmax);
      }
    }
    const bool job = act && !small && (MODE == 1 || need);
    if (act && !job) {
      if (MODE == 3) {
        rec[j] = span_record(a, finish_fit(P, lo, hi, zmax));
      } else {
        const uint32_t w = finish_width(P, lo, hi, zmax);
        if (MODE == 1)
          b[j] = (uint8_t)w;
        else
          mb[j] = w <= bmax ? (uint8_t)w : kNo;
      }
    }
    const uint32_t jobs = __ballot_sync(kFull, job);
    if (jobs) {
      unsigned long long e = 0;
      if (lane == 0) e = atomicAdd(&A.w.cnt[0], (unsigned long long)__popc(jobs));
      e = __shfl_sync(kFull, e, 0) + __popc(jobs & ((1u << lane) - 1u));
      if (job) {
        const bool near = flat && narrow_ref(S.mn) && narrow_diff(S.mx - S.mn);
        put_job(A.w, e, a, N, j, P, bmax, near, MODE != 1);
        if (MODE == 1 && N > kPieceVals) A.w.pieces[atomicAdd(&A.w.cnt[1], 1ull)] = SpanPiece{(uint32_t)e, 0, 0, 1};
      }
    }
    __syncwarp();  // the stage is reused by the next group
  }
}

// One listed partition of the split by a tile of TILE lanes (N = 0: the tile only takes part in the
// warp's steps): moments into the table, line, residual range, width
template <int TILE, typename T>
__device__ __forceinline__ void fit_listed(const SpanArgs<T>& A, uint64_t a, uint32_t N, uint64_t j, uint8_t* __restrict__ b,
                                           uint32_t r) {
  const T* p = A.v + a;
  const bool lin = A.model == LECO_MODEL_LINEAR;
  const int64_t ref = N ? (int64_t)__ldg(p) : 0;
  bool ok = narrow_ref(ref);
  int64_t sum = 0, Sd = 0;
  int32_t mn = INT32_MAX, mx = INT32_MIN;
  const int32_t nm1 = (int32_t)N - 1;
#pragma unroll 4
  for (uint32_t x = r; x < N; x += TILE) {
    const int64_t d = (int64_t)__ldg(p + x) - ref;
    ok = ok && narrow_diff(d);
    const int32_t e = (int32_t)d;
    mn = min(mn, e);
    mx = max(mx, e);
    Sd += e;
    sum += (int64_t)(2 * (int32_t)x - nm1) * e;
  }
  SpanStats S;
  i128 moment;
  const bool near = __all_sync(kFull, ok);
  if (near) {
    mn = tile_min<TILE>(mn);
    mx = tile_max<TILE>(mx);
    Sd = tile_sum<TILE>(Sd);
    sum = tile_sum<TILE>(sum);
    S = stats_from(ref, N, Sd, sum, mn, mx);
    moment = sum;
  } else {
    S = group_stats<TILE>(p, r, N, (uint32_t)TILE);
    moment = line_moment(S, N);
  }
  if (N && r == 0) A.stats[a / kStatVals] = S;
  FitParams P;
  P.B = 0;
  P.fb_shift = 0;
  P.s = 0;
  P.fallback = 0;
  if (N) P = solve_params(lin ? moment : (i128)0, S.mx, S.mn, N, lin);
  int64_t lo = S.mn, hi = S.mx;
  uint64_t zmax = 0;
  if (__any_sync(kFull, N && (lin || P.fallback))) {
    if (__all_sync(kFull, !N || (near && narrow_line(P, N)))) {
      const NarrowLine line(P.B, P.s);
      int32_t l = INT32_MAX, h = INT32_MIN;
      uint64_t G = line.B * r;
      const uint64_t dG = line.B * (uint64_t)TILE;
#pragma unroll 4
      for (uint32_t x = r; x < N; x += TILE, G += dG) {
        const int32_t e = (int32_t)((uint32_t)__ldg(p + x) - (uint32_t)ref) - line.at(G);
        l = min(l, e);
        h = max(h, e);
      }
      lo = ref + tile_min<TILE>(l);
      hi = ref + tile_max<TILE>(h);
    } else {
      lo = INT64_MAX;
      hi = INT64_MIN;
      resid_part(p, r, N, (uint32_t)TILE, P, lo, hi, zmax);
      lo = tile_min<TILE>(lo);
      hi = tile_max<TILE>(hi);
      zmax = tile_max<TILE>(zmax);
    }
  }
  if (N && r == 0) b[j] = (uint8_t)finish_width(P, lo, hi, zmax);
}

// the listed partitions of the split up to kPieceVals values: four at a time, those beyond kTileVals one
// after another
template <typename T>
__global__ void __launch_bounds__(256) k_fit_long(const SpanArgs<T> A, uint8_t* __restrict__ b) {
  const uint64_t nj = *(volatile unsigned long long*)&A.w.cnt[0];
  const uint32_t lane = threadIdx.x & 31u, r = lane & 7u;
  for (uint64_t e0 = ((uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5)) * 4; e0 < nj; e0 += (uint64_t)gridDim.x * 32) {
    const uint64_t e = e0 + (lane >> 3);
    SpanJob q = {};
    if (e < nj) q = A.w.jobs[e];
    fit_listed<8>(A, q.a, q.N <= kTileVals ? q.N : 0u, q.j, b, r);
    uint32_t big = __ballot_sync(kFull, r == 0 && q.N > kTileVals && q.N <= kPieceVals);
    while (big) {
      const int src = __ffs((int)big) - 1;
      big &= big - 1;
      fit_listed<32>(A, __shfl_sync(kFull, q.a, src), __shfl_sync(kFull, q.N, src), __shfl_sync(kFull, q.j, src), b, lane);
    }
  }
}

// ... and those beyond, a CTA each (at most 2^16 values: a split's partition ends with its chunk)
template <typename T>
__global__ void __launch_bounds__(256) k_fit_longest(const SpanArgs<T> A, uint8_t* __restrict__ b) {
  __shared__ SpanStats part[8];
  __shared__ int64_t plo[8], phi[8];
  __shared__ uint64_t pz[8];
  const uint64_t np = *(volatile unsigned long long*)&A.w.cnt[1];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  for (uint64_t k = blockIdx.x; k < np; k += gridDim.x) {
    const SpanJob q = A.w.jobs[A.w.pieces[k].e];
    const T* p = A.v + q.a;
    SpanStats S = group_stats<32>(p, threadIdx.x, q.N, 256);
    if (lane == 0) part[wid] = S;
    __syncthreads();
    S = part[0];
    for (int w = 1; w < 8; w++) {
      S.T0 += part[w].T0;
      S.T1 += part[w].T1;
      S.mn = min(S.mn, part[w].mn);
      S.mx = max(S.mx, part[w].mx);
    }
    if (threadIdx.x == 0) A.stats[q.a / kStatVals] = S;
    const bool lin = A.model == LECO_MODEL_LINEAR;
    const FitParams P = solve_params(lin ? line_moment(S, q.N) : (i128)0, S.mx, S.mn, q.N, lin);
    int64_t lo = S.mn, hi = S.mx;
    uint64_t zmax = 0;
    if (lin || P.fallback) {
      lo = INT64_MAX;
      hi = INT64_MIN;
      resid_part(p, threadIdx.x, q.N, 256, P, lo, hi, zmax);
      lo = tile_min<32>(lo);
      hi = tile_max<32>(hi);
      zmax = tile_max<32>(zmax);
      if (lane == 0) {
        plo[wid] = lo;
        phi[wid] = hi;
        pz[wid] = zmax;
      }
      __syncthreads();
      for (int w = 0; w < 8; w++) {
        lo = min(lo, plo[w]);
        hi = max(hi, phi[w]);
        zmax = max(zmax, pz[w]);
      }
    }
    if (threadIdx.x == 0) b[q.j] = (uint8_t)finish_width(P, lo, hi, zmax);
    __syncthreads();  // the shared parts are reused
  }
}

__device__ __forceinline__ FitParams job_line(const SpanJob& q) {
  FitParams P;
  P.s = q.s;
  P.fallback = q.fallback;
  P.B = q.fallback ? 0 : q.B;
  P.fb_shift = q.fallback ? q.B : 0;
  return P;
}

// Residual range of values x0 + r, + TILE, ... < x1 of a listed span, reduced over the tile. narrow: every
// tile of the warp has a narrow span. CHECK (a warp per span): stops once the range alone needs more than
// bmax bits, first at 32 values spread over a long span (which settles most pairs that do not belong together).
template <int TILE, bool CHECK, typename T>
__device__ __forceinline__ void job_range(const T* __restrict__ p, const SpanJob& q, uint32_t x0, uint32_t x1, uint32_t r,
                                          bool narrow, int64_t& lo, int64_t& hi, uint64_t& zmax) {
  if (narrow) {
    const NarrowLine line(q.B, q.s);
    const uint32_t ref = x0 < x1 ? (uint32_t)__ldg(p) : 0u;
    int32_t l = INT32_MAX, h = INT32_MIN;
    // values xa + r, + TILE, ... < xb, eight loads in flight per lane
    auto pass = [&](uint32_t xa, uint32_t xb) {
      uint64_t G = line.B * (xa + r);
      const uint64_t dG = line.B * (uint64_t)TILE;
      for_runs<TILE, 8>(
          p + xa, xb - xa, r, (T)0,
          [&](T value) {
            const int32_t e = (int32_t)((uint32_t)value - ref) - line.at(G);
            l = min(l, e);
            h = max(h, e);
            G += dG;
          },
          []() { return true; });
    };
    if (CHECK && q.bmax < 31) {
      bool over = false;
      if (x1 - x0 >= 1024) {
        const uint32_t x = x0 + r * ((x1 - x0) >> 5);
        l = h = (int32_t)((uint32_t)__ldg(p + x) - ref) - line.at(line.B * x);
        over = ((uint32_t)tile_max<TILE>(h) - (uint32_t)tile_min<TILE>(l)) >> q.bmax != 0;
      }
      for (uint32_t x = x0; x < x1 && !over; x += 1024) {
        pass(x, min(x + 1024u, x1));
        if (x + 1024 < x1) over = __any_sync(kFull, l <= h && ((uint32_t)h - (uint32_t)l) >> q.bmax != 0);
      }
    } else {
      pass(x0, x1);
    }
    // 32-bit differences from the span's first value: whole again by its 64 bits
    const int64_t ref64 = x0 < x1 ? (int64_t)__ldg(p) : 0;
    lo = ref64 + tile_min<TILE>(l);
    hi = ref64 + tile_max<TILE>(h);
    zmax = 0;
    return;
  }
  const FitParams P = job_line(q);
  lo = INT64_MAX;
  hi = INT64_MIN;
  zmax = 0;
  if (CHECK && q.bmax < 63 && !P.fallback) {
    bool over = false;
    for (uint32_t x = x0; x < x1 && !over; x += 1024) {
      resid_part(p, x + r, min(x + 1024u, x1), (uint32_t)TILE, P, lo, hi, zmax);
      if (x + 1024 < x1) over = __any_sync(kFull, lo <= hi && ((uint64_t)hi - (uint64_t)lo) >> q.bmax != 0);
    }
  } else {
    resid_part(p, x0 + r, x1, (uint32_t)TILE, P, lo, hi, zmax);
  }
  lo = tile_min<TILE>(lo);
  hi = tile_max<TILE>(hi);
  zmax = tile_max<TILE>(zmax);
}

__device__ __forceinline__ void finish_job(const SpanJob& q, int64_t lo, int64_t hi, uint64_t zmax, uint8_t* __restrict__ mb,
                                           Record* __restrict__ rec) {
  const FitParams P = job_line(q);
  if (rec) {
    rec[q.j] = span_record(q.a, finish_fit(P, lo, hi, zmax));
  } else {
    const uint32_t w = finish_width(P, lo, hi, zmax);
    mb[q.j] = w <= q.bmax ? (uint8_t)w : kNo;
  }
}

// Residual ranges of the listed spans under their lines, then the width (mb) or the record (rec): four spans
// of up to kTileVals values per warp at a time, longer ones a warp each, pieces of those beyond kPieceVals. A
// range that rules out a gain may be cut short: the width is at least bitlen(hi - lo) whatever the intercept.
template <typename T>
__global__ void __launch_bounds__(256) k_span_range(const SpanArgs<T> A, uint8_t* __restrict__ mb, Record* __restrict__ rec) {
  const uint64_t nj = *(volatile unsigned long long*)&A.w.cnt[0], np = *(volatile unsigned long long*)&A.w.cnt[1];
  const uint32_t lane = threadIdx.x & 31u, r = lane & 7u;
  const uint64_t gw = (uint64_t)blockIdx.x * 8 + (threadIdx.x >> 5), nw = (uint64_t)gridDim.x * 8;
  for (uint64_t e0 = gw * 4; e0 < nj; e0 += nw * 4) {
    const uint64_t e = e0 + (lane >> 3);
    SpanJob q = {};
    if (e < nj) q = A.w.jobs[e];
    const bool tiled = q.N && q.N <= kTileVals;
    int64_t lo, hi;
    uint64_t zmax;
    if (__any_sync(kFull, tiled)) {
      job_range<8, false>(A.v + q.a, q, 0, tiled ? q.N : 0u, r, __all_sync(kFull, !tiled || q.narrow), lo, hi, zmax);
      if (tiled && r == 0) finish_job(q, lo, hi, zmax, mb, rec);
    }
    uint32_t big = __ballot_sync(kFull, r == 0 && q.N > kTileVals && q.N <= kPieceVals);
    while (big) {
      const int src = __ffs((int)big) - 1;
      big &= big - 1;
      const SpanJob one = A.w.jobs[e0 + (uint64_t)(src >> 3)];
      job_range<32, true>(A.v + one.a, one, 0, one.N, lane, one.narrow != 0, lo, hi, zmax);
      if (lane == 0) finish_job(one, lo, hi, zmax, mb, rec);
    }
  }
  for (uint64_t t = gw; t < np; t += nw) {
    const SpanPiece pc = A.w.pieces[t];
    const SpanJob q = A.w.jobs[pc.e];
    const uint32_t x0 = pc.q * kPieceVals, x1 = min(x0 + kPieceVals, q.N);
    int64_t lo, hi;
    uint64_t zmax;
    job_range<32, true>(A.v + q.a, q, x0, x1, lane, q.narrow != 0, lo, hi, zmax);
    if (lane != 0) continue;
    atomicMin(&A.w.lo[pc.mi], (long long)lo);
    atomicMax(&A.w.hi[pc.mi], (long long)hi);
    atomicMax(&A.w.zmax[pc.mi], (unsigned long long)zmax);
    __threadfence();
    if (atomicAdd(&A.w.done[pc.mi], 1u) + 1u < pc.np) continue;  // the last of the pieces has the whole range
    __threadfence();
    finish_job(q, *(volatile long long*)&A.w.lo[pc.mi], *(volatile long long*)&A.w.hi[pc.mi],
               *(volatile unsigned long long*)&A.w.zmax[pc.mi], mb, rec);
  }
}

// gain of a pair of widths and lengths that merges at width w
__device__ __forceinline__ int64_t gain_of(uint64_t N1, uint32_t b1, uint64_t N2, uint32_t b2, uint32_t w) {
  return (int64_t)(kSmBits + N1 * b1 + N2 * b2) - (int64_t)((N1 + N2) * w);
}

// priority order of two pairs: gain, then the hash of the start, then the smaller start
__device__ __forceinline__ bool beats(int64_t g1, uint64_t s1, int64_t g2, uint64_t s2) {
  if (g1 != g2) return g1 > g2;
  const uint64_t h1 = splitmix64(s1), h2 = splitmix64(s2);
  if (h1 != h2) return h1 > h2;
  return s1 < s2;
}

// Dense rounds: tiles of kMergeTile partitions. k_select: bit j of sel is set when pair j merges (it gains
// and beats both neighbours); the tile's count into cnt.
constexpr uint32_t kMergeTile = 1024;

__global__ void __launch_bounds__(256)
    k_select(const uint64_t* __restrict__ st, const uint8_t* __restrict__ b, const uint8_t* __restrict__ mb, uint64_t m,
             uint32_t* __restrict__ sel, uint64_t* __restrict__ cnt) {
  // [i] belongs to pair base - 1 + i. A pair's gain fits 32 bits (at most 2^24 values of 64 bits); kLoses:
  // it does not merge. Gains tie in most pairs of the first rounds, so each pair's hash is taken once too.
  constexpr int32_t kLoses = INT32_MIN;
  __shared__ uint64_t s_st[kMergeTile + 4], s_hash[kMergeTile + 2];
  __shared__ int32_t s_gain[kMergeTile + 2];
  __shared__ uint8_t s_b[kMergeTile + 4];
  __shared__ uint32_t ws[8];
  const uint64_t base = (uint64_t)blockIdx.x * kMergeTile;
  // all of the tile's loads at once, whether or not a pair turns out to gain, against a
  // chain of loads per pair: 1016 -> 778 us over the rounds of 100M piecewise values (the encode 18.1 -> 17.9 ms)
  constexpr int kPer = (kMergeTile + 4 + 255) / 256;
  uint64_t s0[kPer];
  uint8_t b0[kPer], w0[kPer];
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const uint32_t i = threadIdx.x + 256u * k;
    const uint64_t p = base + i - 1;  // wraps below 0: past every bound
    const bool in = i < kMergeTile + 4;
    s0[k] = in && p <= m ? st[p] : 0;
    b0[k] = in && p < m ? b[p] : 0;
    w0[k] = in && p < m && p + 1 < m ? mb[p] : kNo;
  }
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const uint32_t i = threadIdx.x + 256u * k;
    if (i < kMergeTile + 4) {
      s_st[i] = s0[k];
      s_b[i] = b0[k];
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const uint32_t i = threadIdx.x + 256u * k;
    if (i < kMergeTile + 2) {
      const uint64_t mid = s_st[i + 1];
      s_gain[i] = w0[k] <= 64 ? (int32_t)gain_of(mid - s0[k], b0[k], s_st[i + 2] - mid, s_b[i + 1], w0[k]) : kLoses;
      s_hash[i] = splitmix64(s0[k]);
    }
  }
  __syncthreads();
  uint32_t local = 0;
  for (uint32_t u = threadIdx.x; u < kMergeTile; u += 256) {
    const uint32_t i = u + 1;
    const int32_t g = s_gain[i];
    auto over = [&](uint32_t k) {  // pair i beats pair k
      if (g != s_gain[k]) return g > s_gain[k];
      return s_hash[i] != s_hash[k] ? s_hash[i] > s_hash[k] : s_st[i] < s_st[k];
    };
    const bool ok = g != kLoses && over(i - 1) && over(i + 1);
    const uint32_t w = __ballot_sync(kFull, ok);
    if ((threadIdx.x & 31u) == 0) {
      sel[(base + u) >> 5] = w;
      local += (uint32_t)__popc(w);
    }
  }
  if ((threadIdx.x & 31u) == 0) ws[threadIdx.x >> 5] = local;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; k++) local += ws[k];
    cnt[blockIdx.x] = local;
  }
}

// the moments of two partitions [a, mid), [mid, c) that merge, where the result carries them
template <typename T>
__device__ __forceinline__ void merge_stats(const T* __restrict__ v, SpanStats* __restrict__ stats, uint64_t a,
                                            uint64_t mid, uint64_t c) {
  if (c - a <= kStatVals) return;
  stats[a / kStatVals] = combine_stats(part_stats(v, a, (uint32_t)(mid - a), stats), mid - a,
                                       part_stats(v, mid, (uint32_t)(c - mid), stats));
}

// The moments of the partitions that the chosen pairs make, where those carry them, by a warp per 32 pairs:
// the values of parts without moments are staged together as 32-bit differences, from the first merging lane's
// start to the last one's end, instead of each lane walking its own. A kernel of its own, with the starts of
// its next pairs in flight, which leaves k_compact few registers and its loads all at once: over the rounds
// of 100M piecewise values 2.1 + 0.6 ms, against 3.46 ms for both in one kernel (the encode 19.4 -> 18.95 ms).
template <typename T>
__global__ void __launch_bounds__(kSpanBlock, 8)
    k_merge_stats(const T* __restrict__ v, const uint64_t* __restrict__ st, uint64_t m, const uint32_t* __restrict__ sel,
                  SpanStats* __restrict__ stats) {
  __shared__ int32_t raw[kSpanBlock / 32][kSpanStage];
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  int32_t* stage = raw[wib];
  const uint64_t words = (m + 31) / 32, gw = (uint64_t)gridDim.x * (kSpanBlock / 32);
  // the starts of the next 32 pairs are on their way while this one's are looked at: most rounds merge few
  // pairs that carry moments, and are these loads
  uint64_t g = (uint64_t)blockIdx.x * (kSpanBlock / 32) + wib;
  uint32_t wn = 0;
  uint64_t sn = 0, xn = 0;
  auto fetch = [&](uint64_t at) {
    if (at >= words) return;
    const uint64_t p = at * 32 + lane;
    wn = sel[at];
    sn = st[p < m ? p : m];
    if (lane < 2) xn = st[p + 32 < m ? p + 32 : m];
  };
  fetch(g);
  for (; g < words; g += gw) {
    const uint32_t w = wn;
    const uint64_t a = sn, x = xn;
    fetch(g + gw);
    if (w == 0) continue;
    const bool chosen = (w >> lane) & 1u;
    uint64_t mid = __shfl_down_sync(kFull, a, 1), c = __shfl_down_sync(kFull, a, 2);
    const uint64_t x0 = __shfl_sync(kFull, x, 0), xl = __shfl_sync(kFull, x, lane & 1u);
    if (lane == 31) mid = x0;
    if (lane >= 30) c = xl;
    const bool need = chosen && c - a > kStatVals;
    const bool left = need && mid - a <= kStatVals, right = need && c - mid <= kStatVals;  // parts without moments
    const uint32_t lanes = __ballot_sync(kFull, left || right);
    if (!__any_sync(kFull, need)) continue;
    SpanStats L, R;  // the other parts' loads go out first
    if (need && !left) L = stats[a / kStatVals];
    if (need && !right) R = stats[mid / kStatVals];
    int64_t ref = 0;
    uint64_t ga = 0;
    bool narrow = false;
    if (lanes) {
      ga = __shfl_sync(kFull, left ? a : mid, __ffs((int)lanes) - 1);
      const uint64_t gc = __shfl_sync(kFull, right ? c : mid, 31 - __clz((int)lanes));
      if (gc - ga <= kSpanStage) {
        ref = (int64_t)__ldg(v + ga);
        bool ok = narrow_ref(ref);
#pragma unroll 4
        for (uint32_t t = lane; t < (uint32_t)(gc - ga); t += 32) {
          const int64_t d = (int64_t)__ldg(v + ga + t) - ref;
          ok = ok && narrow_diff(d);
          stage[t] = (int32_t)d;
        }
        narrow = __all_sync(kFull, ok);
        __syncwarp();
      }
    }
    auto part = [&](uint64_t from, uint32_t N) -> SpanStats {
      if (!narrow) return lane_stats(v + from, N);
      const int32_t* dp = stage + (uint32_t)(from - ga);
      int64_t sum = 0, Sd = 0;
      int32_t mn = INT32_MAX, mx = INT32_MIN, u = 1 - (int32_t)N;
#pragma unroll 4
      for (uint32_t x = 0; x < N; x++, u += 2) {
        const int32_t d = dp[x];
        mn = min(mn, d);
        mx = max(mx, d);
        sum += (int64_t)u * d;
        Sd += d;
      }
      return stats_from(ref, N, Sd, sum, mn, mx);
    };
    if (left) L = part(a, (uint32_t)(mid - a));
    if (right) R = part(mid, (uint32_t)(c - mid));
    if (need) stats[a / kStatVals] = combine_stats(L, mid - a, R);
    __syncwarp();  // the stage is reused
  }
}

// The next round's partitions. Partition p survives unless pair p - 1 merges; its rank is p less the pairs
// that merge before pair p - 1.
__global__ void __launch_bounds__(256)
    k_compact(const uint64_t* __restrict__ st, const uint8_t* __restrict__ b, const uint8_t* __restrict__ mb, uint64_t m,
              const uint32_t* __restrict__ sel, const uint64_t* __restrict__ before, const uint64_t* __restrict__ total,
              uint64_t* __restrict__ nst, uint8_t* __restrict__ nb, uint8_t* __restrict__ nmb) {
  __shared__ uint32_t bits[kMergeTile / 32 + 2];  // word i: pairs base - 32 + 32 i ..
  __shared__ uint32_t pre[kMergeTile / 32];       // pairs of the tile that merge before word i
  const uint64_t base = (uint64_t)blockIdx.x * kMergeTile, words = (m + 31) / 32;
  const uint32_t t = threadIdx.x;
  // the tile's partitions, all loads at once
  constexpr int kPer = kMergeTile / 256;
  uint64_t s0[kPer];
  uint8_t b0[kPer], w0[kPer];
#pragma unroll
  for (int k = 0; k < kPer; k++) {
    const uint64_t p = base + t + 256u * k;
    s0[k] = p <= m ? st[p] : 0;
    b0[k] = p < m ? b[p] : 0;
    w0[k] = p + 1 < m ? mb[p] : 0;
  }
  if (t < kMergeTile / 32 + 2) {
    const int64_t w = (int64_t)(base >> 5) - 1 + (int64_t)t;
    bits[t] = w >= 0 && (uint64_t)w < words ? sel[w] : 0u;
  }
  __syncthreads();
  if (t < 32) {
    const uint32_t c = (uint32_t)__popc(bits[t + 1]);
    uint32_t inc = c;
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, inc, o);
      if (t >= o) inc += y;
    }
    pre[t] = inc - c;
  }
  __syncthreads();
  auto merges = [&](uint32_t i) -> bool {  // pair base - 32 + i
    return (bits[i >> 5] >> (i & 31u)) & 1u;
  };
  const uint64_t merged = before[blockIdx.x];
#pragma unroll
  for (int r = 0; r < kPer; r++) {
    const uint32_t u = t + 256u * r, i = u + 32u;
    const uint64_t p = base + u;
    if (p >= m || merges(i - 1u)) continue;  // past the end, or absorbed
    const bool mp = merges(i);
    const uint64_t k = p - (merged + pre[u >> 5] + (uint32_t)__popc(bits[i >> 5] & ((1u << (u & 31u)) - 1u)));
    nst[k] = s0[r];
    nb[k] = mp ? w0[r] : b0[r];
    // the next survivor is q; the pair of the two is new when either of them is
    const uint32_t qi = i + (mp ? 2u : 1u);
    const uint64_t q = p + (mp ? 2 : 1);
    if (q < m) nmb[k] = mp || merges(qi) ? kDirty : w0[r];
    if (p == 0) nst[m - *total] = st[m];
  }
}

// ------------------------------------------------------------------------------ sparse rounds
//
// The partitions keep their slots (the indexes at the switch); left / right link the live ones. A round:
// k_sparse_select takes the candidate pairs (left partitions whose pair gains; once each, by `seen`),
// lists the ones that beat both neighbours and keeps the others as candidates; k_sparse_apply merges
// them; k_sparse_plan fits the pairs that changed (short ones at once, the others through the job list) and
// adds them to the candidates; k_span_range ends the fits. Every list's length stays on the device, in
// a counter per round.
struct Sparse {
  uint64_t n;
  const uint64_t* st;
  uint8_t *b, *mb;
  uint32_t *left, *right, *seen, *merged;
  uint32_t* chosen;
};
struct SparseRound {
  unsigned long long cands, chosen, jobs, pieces, slots;
};

__global__ void k_sparse_init(Sparse S, uint64_t m, uint32_t* __restrict__ cand, SparseRound* __restrict__ r) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < m; j += (uint64_t)gridDim.x * blockDim.x) {
    S.left[j] = j ? (uint32_t)(j - 1) : kSlotEnd;
    S.right[j] = j + 1 < m ? (uint32_t)(j + 1) : kSlotEnd;
    S.seen[j] = 0;
    S.merged[j] = 0;
    if (j + 1 == m) S.mb[j] = kNo;
    if (j + 1 < m && S.mb[j] <= 64) cand[atomicAdd(&r->cands, 1ull)] = (uint32_t)j;
  }
}

__device__ __forceinline__ uint64_t slot_end(const Sparse& S, uint32_t j) {
  const uint32_t r = S.right[j];
  return r == kSlotEnd ? S.n : S.st[r];
}

// gain of the pair of slot j and its right neighbour (mb[j] <= 64)
__device__ __forceinline__ int64_t slot_gain(const Sparse& S, uint32_t j) {
  const uint32_t r = S.right[j];
  const uint64_t mid = S.st[r];
  return gain_of(mid - S.st[j], S.b[j], slot_end(S, r) - mid, S.b[r], S.mb[j]);
}

__global__ void k_sparse_select(Sparse S, uint32_t round, const uint32_t* __restrict__ cand, SparseRound* __restrict__ r,
                                uint32_t* __restrict__ next, SparseRound* __restrict__ rn) {
  const uint64_t nc = r->cands;
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < nc; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t j = cand[t];
    if (S.mb[j] > 64 || atomicExch(&S.seen[j], round) == round) continue;
    const uint64_t a = S.st[j];
    const int64_t g = slot_gain(S, j);
    const uint32_t l = S.left[j], rt = S.right[j];
    bool ok = l == kSlotEnd || S.mb[l] > 64 || beats(g, a, slot_gain(S, l), S.st[l]);
    if (ok && S.mb[rt] <= 64) ok = beats(g, a, slot_gain(S, rt), S.st[rt]);
    if (ok)
      S.chosen[atomicAdd(&r->chosen, 1ull)] = j;
    else
      next[atomicAdd(&rn->cands, 1ull)] = j;
  }
}

template <typename T>
__global__ void k_sparse_apply(Sparse S, const T* __restrict__ v, SpanStats* __restrict__ stats, uint32_t round,
                               const SparseRound* __restrict__ r) {
  const uint64_t nc = r->chosen;
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < nc; t += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t j = S.chosen[t], q = S.right[j], qq = S.right[q];
    merge_stats(v, stats, S.st[j], S.st[q], qq == kSlotEnd ? S.n : S.st[qq]);
    S.b[j] = S.mb[j];
    S.right[j] = qq;
    if (qq != kSlotEnd) S.left[qq] = j;
    S.mb[q] = kDead;
    S.merged[j] = round;
  }
}

// the two pairs of every partition merged this round (the left one is its left neighbour's own when that
// merged too)
template <typename T>
__global__ void k_sparse_plan(Sparse S, const SpanArgs<T> A, uint32_t round, const SparseRound* __restrict__ r,
                              uint32_t* __restrict__ next, SparseRound* __restrict__ rn) {
  const uint64_t nc = 2 * r->chosen;
  for (uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; t < nc; t += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t j = S.chosen[t >> 1];
    if (t & 1) {
      j = S.left[j];
      if (j == kSlotEnd || S.merged[j] == round) continue;
    }
    const uint32_t q = S.right[j];
    if (q == kSlotEnd) {
      S.mb[j] = kNo;
      continue;
    }
    const uint64_t a = S.st[j], mid = S.st[q], c = slot_end(S, q);
    if (c - a > A.cap) {
      S.mb[j] = kNo;
      continue;
    }
    const uint32_t N = (uint32_t)(c - a);
    const bool lin = A.model == LECO_MODEL_LINEAR;
    const SpanStats M = combine_stats(part_stats(A.v, a, (uint32_t)(mid - a), A.stats), mid - a,
                                      part_stats(A.v, mid, (uint32_t)(c - mid), A.stats));
    const FitParams P = solve_params(lin ? line_moment(M, N) : (i128)0, M.mx, M.mn, N, lin);
    const uint32_t bmax = gain_width((uint32_t)(mid - a), S.b[j], (uint32_t)(c - mid), S.b[q]);
    if (N > kLaneVals && (lin || P.fallback)) {
      const bool near = narrow_line(P, N) && narrow_ref(M.mn) && narrow_diff(M.mx - M.mn);
      put_job(A.w, atomicAdd(&A.w.cnt[0], 1ull), a, N, j, P, bmax, near, true);
    } else {
      int64_t lo = M.mn, hi = M.mx;
      uint64_t zmax = 0;
      if (lin || P.fallback) {
        lo = INT64_MAX;
        hi = INT64_MIN;
        resid_part(A.v + a, 0, N, 1, P, lo, hi, zmax);
      }
      const uint32_t w = finish_width(P, lo, hi, zmax);
      S.mb[j] = w <= bmax ? (uint8_t)w : kNo;
    }
    next[atomicAdd(&rn->cands, 1ull)] = j;
  }
}

// live slots as bits, and their number per tile; then the surviving starts side by side
__global__ void __launch_bounds__(256) k_live(const uint8_t* __restrict__ mb, uint64_t m, uint32_t* __restrict__ live,
                                              uint64_t* __restrict__ cnt) {
  __shared__ uint32_t total;
  if (threadIdx.x == 0) total = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kMergeTile;
  for (uint32_t u = threadIdx.x; u < kMergeTile; u += 256) {
    const uint64_t p = base + u;
    const uint32_t w = __ballot_sync(kFull, p < m && mb[p] != kDead);
    if ((threadIdx.x & 31u) == 0) {
      live[p >> 5] = w;
      atomicAdd(&total, (uint32_t)__popc(w));
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) cnt[blockIdx.x] = total;
}

__global__ void __launch_bounds__(256)
    k_gather_live(const uint64_t* __restrict__ st, uint64_t m, uint64_t n, const uint32_t* __restrict__ live,
                  const uint64_t* __restrict__ before, const uint64_t* __restrict__ total, uint64_t* __restrict__ nst) {
  __shared__ uint32_t pre[kMergeTile / 32];
  const uint64_t base = (uint64_t)blockIdx.x * kMergeTile;
  const uint32_t t = threadIdx.x;
  if (t < 32) {
    const uint32_t c = (uint32_t)__popc(live[(base >> 5) + t]);
    uint32_t inc = c;
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(kFull, inc, o);
      if (t >= o) inc += y;
    }
    pre[t] = inc - c;
  }
  __syncthreads();
  for (uint32_t u = t; u < kMergeTile; u += 256) {
    const uint64_t p = base + u;
    if (p >= m) break;
    const uint32_t w = live[p >> 5];
    if ((w >> (u & 31u)) & 1u) nst[before[blockIdx.x] + pre[u >> 5] + (uint32_t)__popc(w & ((1u << (u & 31u)) - 1u))] = st[p];
    if (p == 0) nst[*total] = n;
  }
}

template <typename T>
cudaError_t dalloc(T** p, uint64_t elems, cudaStream_t st) {
  return dev_alloc((void**)p, (elems ? elems : 1) * sizeof(T), st);
}

// the split into bitmap; seeds (nullptr: the plain split) is scratch for the chunks' seeds
template <typename T>
cudaError_t launch_split(const T* v, uint64_t n, uint64_t nchunks, uint32_t cap, int64_t tfloor, uint64_t* seeds,
                         uint64_t* bitmap, cudaStream_t st) {
  if (seeds) {
    k_chunk_seed<<<grid_for(nchunks, 1, 8), 256, 0, st>>>(v, n, seeds);
    k_split<T, true><<<(unsigned)(2 * nchunks), kSplitThreads, 0, st>>>(v, n, cap, tfloor, seeds, bitmap);
  } else {
    k_split<T, false><<<(unsigned)nchunks, kSplitThreads, 0, st>>>(v, n, cap, tfloor, nullptr, bitmap);
  }
  return cudaGetLastError();
}

// one allocation handed out in 256-byte steps: sized by a first pass over the same calls with no base
struct Arena {
  char* base = nullptr;
  uint64_t used = 0;
  template <typename U>
  U* take(uint64_t elems) {
    U* p = base ? reinterpret_cast<U*>(base + used) : nullptr;
    used += (elems * sizeof(U) + 255) & ~255ull;
    return p;
  }
};

constexpr uint32_t kSparseRounds = 6;  // sparse rounds between two looks at the count of merges

// the merge from the split's m partitions in starts_out: rounds until none merges; m starts (and n) in
// starts_out, and the records of their fits when rec_out is given
template <typename T>
cudaError_t merge_rounds(const T* v, uint64_t n, uint32_t cap, int model, uint64_t* starts_out, uint64_t m,
                         uint64_t* m_out, Record** rec_out, cudaStream_t s) {
  const uint64_t tiles = (m + kMergeTile - 1) / kMergeTile, spans = 2 * n / kPieceVals + 2;
  SpanArgs<T> A;
  A.v = v;
  A.cap = cap;
  A.model = model;
  uint64_t *st_b, *cnt, *before, *scan, *total;
  uint8_t *b_a, *b_b, *mb_a, *mb_b;
  uint32_t* sel;
  auto layout = [&](Arena& ar) {
    A.stats = ar.take<SpanStats>(n / kStatVals + 1);
    st_b = ar.take<uint64_t>(m + 1);
    b_a = ar.take<uint8_t>(m);
    b_b = ar.take<uint8_t>(m);
    mb_a = ar.take<uint8_t>(m);
    mb_b = ar.take<uint8_t>(m);
    sel = ar.take<uint32_t>(tiles * (kMergeTile / 32));
    cnt = ar.take<uint64_t>(tiles);
    before = ar.take<uint64_t>(tiles);
    scan = ar.take<uint64_t>(tiles / 2048 + 3);
    total = ar.take<uint64_t>(1);
    A.w.jobs = ar.take<SpanJob>(2 * n / kLaneVals + 2);  // spans beyond kLaneVals in pairs cover n twice at most
    A.w.pieces = ar.take<SpanPiece>(2 * spans);
    A.w.lo = ar.take<long long>(spans);
    A.w.hi = ar.take<long long>(spans);
    A.w.zmax = ar.take<unsigned long long>(spans);
    A.w.done = ar.take<uint32_t>(spans);
    A.w.cnt = ar.take<unsigned long long>(3);
  };
  Arena ar;
  layout(ar);
  cudaError_t e = dev_alloc((void**)&ar.base, ar.used, s);
  if (e != cudaSuccess) return e;
  ar.used = 0;
  layout(ar);
  char *arena = ar.base, *sparse_arena = nullptr;
  const int wide = sm_count() * 8;
  // groups of 32 spans differ in work a hundredfold (none dirty to all solved): an eighth of the strided
  // share per warp lets the scheduler even them out, 18.6 -> 18.1 ms for 100M piecewise values against 8 CTAs
  // per SM; a group per warp pays for the CTAs (18.7)
  auto span_grid = [&](uint64_t count) { return grid_for((count + 31) / 32, kSpanBlock / 32, 64); };
  auto clear = [&]() { return cudaMemsetAsync(A.w.cnt, 0, 3 * sizeof(unsigned long long), s); };
  uint64_t *cur = starts_out, *nxt = st_b;
  e = clear();
  if (e == cudaSuccess) {
    k_fit_spans<T, 1><<<span_grid(m), kSpanBlock, 0, s>>>(A, cur, m, b_a, nullptr, nullptr);
    k_fit_long<T><<<wide, 256, 0, s>>>(A, b_a);
    k_fit_longest<T><<<sm_count() * 2, 256, 0, s>>>(A, b_a);
    e = cudaMemsetAsync(mb_a, kDirty, m, s);
  }
  bool sparse = false;
  while (e == cudaSuccess && m > 1) {
    e = clear();
    if (e != cudaSuccess) break;
    k_fit_spans<T, 2><<<span_grid(m - 1), kSpanBlock, 0, s>>>(A, cur, m - 1, b_a, mb_a, nullptr);
    k_span_range<T><<<wide, 256, 0, s>>>(A, mb_a, nullptr);
    e = cudaGetLastError();
    sparse = sparse || m <= kSparseBelow;
    if (e != cudaSuccess || sparse) break;
    const uint64_t nt = (m + kMergeTile - 1) / kMergeTile;
    k_select<<<(unsigned)nt, 256, 0, s>>>(cur, b_a, mb_a, m, sel, cnt);
    e = scan_u64(cnt, nt, before, scan, total, s);
    uint64_t merges = 0;
    if (e == cudaSuccess) e = cudaMemcpyAsync(&merges, total, 8, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess || merges == 0) break;
    k_merge_stats<T><<<span_grid(m), kSpanBlock, 0, s>>>(v, cur, m, sel, A.stats);
    k_compact<<<(unsigned)nt, 256, 0, s>>>(cur, b_a, mb_a, m, sel, before, total, nxt, b_b, mb_b);
    e = cudaGetLastError();
    std::swap(cur, nxt);
    std::swap(b_a, b_b);
    std::swap(mb_a, mb_b);
    sparse = merges * kSparseShare < m && m < kSlotEnd;
    m -= merges;
  }
  if (e == cudaSuccess && sparse) {
    Sparse S;
    S.n = n;
    S.st = cur;
    S.b = b_a;
    S.mb = mb_a;
    uint32_t *cand[2];
    SparseRound* rounds[2];
    auto slots = [&](Arena& a2) {
      S.left = a2.take<uint32_t>(m);
      S.right = a2.take<uint32_t>(m);
      S.seen = a2.take<uint32_t>(m);
      S.merged = a2.take<uint32_t>(m);
      S.chosen = a2.take<uint32_t>(m);
      cand[0] = a2.take<uint32_t>(2 * m);  // a slot enters at most once from each of two kernels
      cand[1] = a2.take<uint32_t>(2 * m);
      rounds[0] = a2.take<SparseRound>(kSparseRounds + 1);
      rounds[1] = a2.take<SparseRound>(kSparseRounds + 1);
    };
    Arena a2;
    slots(a2);
    e = dev_alloc((void**)&a2.base, a2.used, s);
    a2.used = 0;
    slots(a2);
    sparse_arena = a2.base;
    const uint64_t round_bytes = sizeof(SparseRound) * (kSparseRounds + 1);
    const int grid = grid_for(m, 256, 2);
    if (e == cudaSuccess) e = cudaMemsetAsync(rounds[0], 0, round_bytes, s);
    if (e == cudaSuccess) k_sparse_init<<<grid_for(m, 256, 8), 256, 0, s>>>(S, m, cand[0], rounds[0]);
    uint32_t round = 1;
    int side = 0;
    for (unsigned long long merges = 1; e == cudaSuccess && merges; side ^= 1) {
      SparseRound* r = rounds[side];
      for (uint32_t k = 0; k < kSparseRounds; k++, round++) {
        uint32_t *c = cand[round & 1u ? 0 : 1], *next = cand[round & 1u ? 1 : 0];
        SpanArgs<T> B = A;
        B.w.cnt = &r[k].jobs;
        k_sparse_select<<<grid, 256, 0, s>>>(S, round, c, r + k, next, r + k + 1);
        k_sparse_apply<T><<<grid, 256, 0, s>>>(S, v, A.stats, round, r + k);
        k_sparse_plan<T><<<grid, 256, 0, s>>>(S, B, round, r + k, next, r + k + 1);
        k_span_range<T><<<sm_count() * 4, 256, 0, s>>>(B, S.mb, nullptr);
      }
      e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaMemcpyAsync(&merges, &r[kSparseRounds - 1].chosen, 8, cudaMemcpyDeviceToHost, s);
      SparseRound* rn = rounds[side ^ 1];
      if (e == cudaSuccess) e = cudaMemsetAsync(rn, 0, round_bytes, s);
      if (e == cudaSuccess)
        e = cudaMemcpyAsync(&rn->cands, &r[kSparseRounds].cands, 8, cudaMemcpyDeviceToDevice, s);
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    }
    if (e == cudaSuccess) {  // the live slots' starts side by side
      const uint64_t nt = (m + kMergeTile - 1) / kMergeTile;
      k_live<<<(unsigned)nt, 256, 0, s>>>(mb_a, m, sel, cnt);
      e = scan_u64(cnt, nt, before, scan, total, s);
      if (e == cudaSuccess) {
        k_gather_live<<<(unsigned)nt, 256, 0, s>>>(cur, m, n, sel, before, total, nxt);
        e = cudaMemcpyAsync(&m, total, 8, cudaMemcpyDeviceToHost, s);
      }
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      std::swap(cur, nxt);
    }
  }
  if (e == cudaSuccess && rec_out) {
    e = dalloc(rec_out, m, s);  // the final partitions' fits
    if (e == cudaSuccess) e = clear();
    if (e == cudaSuccess) {
      k_fit_spans<T, 3><<<span_grid(m), kSpanBlock, 0, s>>>(A, cur, m, nullptr, nullptr, *rec_out);
      k_span_range<T><<<wide, 256, 0, s>>>(A, nullptr, *rec_out);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess && cur != starts_out)
    e = cudaMemcpyAsync(starts_out, cur, (m + 1) * 8, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFreeAsync(arena, s);
  if (sparse_arena) cudaFreeAsync(sparse_arena, s);
  if (e != cudaSuccess && rec_out && *rec_out) {
    cudaFreeAsync(*rec_out, s);
    *rec_out = nullptr;
  }
  if (e == cudaSuccess) *m_out = m;
  return e;
}

}  // namespace


// Fixed partition-size search (§3.2.1), in the reading the oracle states (R9): SplitMix64-placed
// sample subsequences, an exponential phase over powers of two that ends after the first size above
// its predecessor's, then a back search with halving steps, stopping when a move gains < 0.01 %.
cudaError_t search_partition_size(const void* values, int dtype, uint64_t n, int model, uint32_t N, double frac,
                                  uint64_t seed, uint32_t* best_L, uint64_t* best_bits, uint64_t* evals,
                                  cudaStream_t st) {
  *best_L = 1;
  *best_bits = 0;
  *evals = 0;
  if (n == 0) return cudaSuccess;
  if (n < N) N = (uint32_t)n;
  std::vector<uint64_t> h_starts;
  if (n <= N) {
    h_starts.push_back(0);
  } else {
    uint64_t k = (uint64_t)(frac * (double)n / (double)N);
    if (k < 1) k = 1;
    for (uint64_t i = 0; i < k; i++) h_starts.push_back(splitmix64(seed + i) % (n - N + 1));
  }
  const uint64_t k = h_starts.size();
  uint64_t* d_starts = nullptr;
  unsigned long long* d_total = nullptr;
  cudaError_t e = dalloc(&d_starts, k, st);
  if (e == cudaSuccess) e = dalloc(&d_total, 1, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d_starts, h_starts.data(), 8 * k, cudaMemcpyHostToDevice, st);
  std::map<uint32_t, uint64_t> cache;
  auto size_at = [&](uint32_t L) -> uint64_t {
    auto it = cache.find(L);
    if (it != cache.end()) return it->second;
    unsigned long long total = 0;
    if (e == cudaSuccess) e = cudaMemsetAsync(d_total, 0, 8, st);
    const uint64_t parts = k * ((N + L - 1) / L);
    if (e == cudaSuccess) {
      if (L <= kTinySpan)
        k_sample_sizes_thread<<<grid_for(parts, 256, 8), 256, 0, st>>>(values, dtype, d_starts, k, N, L, model, d_total);
      else
        k_sample_sizes_warp<<<grid_for(parts * 32, 256, 8), 256, 0, st>>>(values, dtype, d_starts, k, N, L, model,
                                                                          d_total);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&total, d_total, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cache[L] = total;
    return total;
  };
  uint32_t best = 1;
  uint64_t best_s = size_at(1), prev_s = best_s;
  for (uint64_t L = 2; e == cudaSuccess; L *= 2) {  // exponential phase
    const uint32_t LL = (uint32_t)(L < N ? L : N);
    const uint64_t s = size_at(LL);
    if (s < best_s) {
      best_s = s;
      best = LL;
    }
    if (s > prev_s || LL == N) break;
    prev_s = s;
  }
  for (uint32_t step = best / 2; step > 0 && e == cudaSuccess;) {  // back search
    uint32_t cand = best;
    uint64_t cand_s = best_s;
    if (best > step) {
      const uint64_t s = size_at(best - step);
      if (s < cand_s) {
        cand_s = s;
        cand = best - step;
      }
    }
    if (best + step <= N) {
      const uint64_t s = size_at(best + step);
      if (s < cand_s) {
        cand_s = s;
        cand = best + step;
      }
    }
    if (cand == best) {
      step /= 2;
      continue;
    }
    const bool small_gain = (best_s - cand_s) * 10000 < best_s;
    best = cand;
    best_s = cand_s;
    if (small_gain) break;
  }
  if (d_starts) cudaFreeAsync(d_starts, st);
  if (d_total) cudaFreeAsync(d_total, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) {
    *best_L = best;
    *best_bits = best_s;
    *evals = cache.size();
  }
  return e;
}

// Runs split + merge; writes m+1 starts to starts_out (capacity n+1) and m to *m_out. rec_out:
// when non-null, receives m records (a new device allocation from the library pool; the caller
// frees it) holding the full fit of every final partition, as the encoder's fit writes them.
cudaError_t var_partition_fit(const void* values, int dtype, uint64_t n, double tau, uint32_t cap, int model,
                              bool seeded, uint64_t* starts_out, uint64_t* m_out, Record** rec_out, cudaStream_t st) {
  *m_out = 0;
  if (rec_out) *rec_out = nullptr;
  if (n == 0) {
    const uint64_t zero = 0;
    cudaError_t e = cudaMemcpyAsync(starts_out, &zero, 8, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    return e;
  }
  const bool u32 = dtype == LECO_U32;
  const double thresh = tau * (double)kSmBits;
  const uint64_t nw = (n + 63) / 64;
  const uint64_t nchunks = (n + kChunk - 1) / kChunk;
  // C <= tau * S_M for an integer C: C <= floor(tau * S_M) (thresh >= 0, below 2^62 here)
  const int64_t tfloor = thresh < 4.0e18 ? (int64_t)floor(thresh) : INT64_MAX;
  uint64_t m = 0;
  cudaError_t e = cudaSuccess;
  {  // split
    uint64_t *bitmap = nullptr, *cnt = nullptr, *pos = nullptr, *scan_scratch = nullptr, *d_total = nullptr;
    uint64_t* seeds = nullptr;
    const uint64_t scan_elems = nchunks / 2048 + 2;
    if (e == cudaSuccess) e = dalloc(&bitmap, nw, st);
    if (e == cudaSuccess) e = dalloc(&cnt, nchunks, st);
    if (e == cudaSuccess) e = dalloc(&pos, nchunks, st);
    if (e == cudaSuccess) e = dalloc(&scan_scratch, scan_elems + 1, st);
    if (e == cudaSuccess) e = dalloc(&d_total, 1, st);
    if (e == cudaSuccess && seeded) {
      e = dalloc(&seeds, nchunks, st);
      if (e == cudaSuccess) e = cudaMemsetAsync(bitmap, 0, 8 * nw, st);
    }
    if (e == cudaSuccess)
      e = u32 ? launch_split(static_cast<const uint32_t*>(values), n, nchunks, cap, tfloor, seeds, bitmap, st)
              : launch_split(static_cast<const uint64_t*>(values), n, nchunks, cap, tfloor, seeds, bitmap, st);
    if (e == cudaSuccess) {
      k_count_starts<<<(unsigned)nchunks, 256, 0, st>>>(bitmap, nw, cnt);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = scan_u64(cnt, nchunks, pos, scan_scratch, d_total, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(&m, d_total, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) {
      k_scatter_starts<<<(unsigned)nchunks, 256, 0, st>>>(bitmap, nw, pos, n, m, starts_out);
      e = cudaGetLastError();
    }
    for (uint64_t* p : {bitmap, cnt, pos, scan_scratch, d_total, seeds})
      if (p) cudaFreeAsync(p, st);
  }
  if (e != cudaSuccess) return e;

  return u32 ? merge_rounds(static_cast<const uint32_t*>(values), n, cap, model, starts_out, m, m_out, rec_out, st)
             : merge_rounds(static_cast<const uint64_t*>(values), n, cap, model, starts_out, m, m_out, rec_out, st);
}

cudaError_t var_partition(const void* values, int dtype, uint64_t n, double tau, uint32_t cap, int model, bool seeded,
                          uint64_t* starts_out, uint64_t* m_out, cudaStream_t st) {
  return var_partition_fit(values, dtype, n, tau, cap, model, seeded, starts_out, m_out, nullptr, st);
}

namespace {
// lenbits[p] = len_p * b_p and the widest b, from records whose fits are done (variable partitions)
__global__ void k_lenbits(const Record* __restrict__ rec, const uint64_t* __restrict__ starts, uint64_t m,
                          uint64_t* __restrict__ lenbits, uint32_t* __restrict__ max_b) {
  uint32_t mb = 0;
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m; p += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t b = w3_b(rec[p].word3);
    lenbits[p] = (starts[p + 1] - starts[p]) * b;
    mb = max(mb, b);
  }
  for (int o = 16; o > 0; o >>= 1) mb = max(mb, __shfl_down_sync(kFull, mb, o));
  if ((threadIdx.x & 31u) == 0 && mb) atomicMax(max_b, mb);
}
}  // namespace

cudaError_t launch_lenbits(const Record* rec, const uint64_t* starts, uint64_t m, uint64_t* lenbits, uint32_t* max_b,
                           cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(max_b, 0, sizeof(uint32_t), st);
  if (e != cudaSuccess || m == 0) return e;
  k_lenbits<<<grid_for(m, 256, 8), 256, 0, st>>>(rec, starts, m, lenbits, max_b);
  return cudaGetLastError();
}

}  // namespace leco

