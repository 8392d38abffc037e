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
constexpr uint64_t kNone = ~0ull;  // no merged size (pair longer than the cap)

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
// The moments of a span's values (w = the value as two's complement int64, x = the local index):
// T0 = sum w, T1 = sum x w, and min and max of w. Two adjacent spans' moments combine exactly (the
// right span's x shifts by the left span's length: T1 gains N_left T0_right), and they give the
// least-squares moment S = sum (2x - (N-1)) w = 2 T1 - (N-1) T0 of the fit and its bounds, so a
// refit needs one pass over the values: the residual range under the snapped line (none for the
// constant model, whose residuals are the values themselves). The moments move with the partitions
// when a round compacts them (a merged pair's are combined then), and the final partitions' fits
// are taken once, from their moments, at the end.
// a pair too long for one warp: its residual range is reduced over pieces of kPiece values
struct LongPair {
  uint64_t j;  // pair index
  uint64_t k;  // slot of its left partition
  uint64_t a;  // first position
  FitParams P;
  uint32_t N;
  uint32_t pad;
};

constexpr uint32_t kTinySpan = 256;    // size search: a thread per sampled partition up to this size
constexpr uint32_t kWarpSpan = 4096;   // a warp fits longer pairs up to this long (split partitions: any)
constexpr uint32_t kPiece = 2048;      // values per piece of a longer pair
constexpr int kGroupBlock = 256;       // 8 warps, each taking 32 spans at a time
constexpr uint32_t kStageBytes = 4096; // per warp: a group's values are staged when they fit

struct MergeWork {
  LongPair* longs;
  uint64_t* pieces;
  unsigned long long* counters;  // [long pairs, pieces]
  long long* lo;                 // per long pair
  long long* hi;
  unsigned long long* zmax;
};

// Full fits of spans. MODE 1: every partition of the split (its moments from a pass over its
// values, into stats[j]; size S_M + len * b into size_out[j]). MODE 2: the dirty adjacent pairs
// [st[j], st[j + 2)) (moments combined from stats[j] and stats[j + 1]; merged size into
// size_out[j]). MODE 3: the final partitions (moments stats[j]; record into rec[j], as the
// encoder's fit writes it). A warp takes 32 consecutive spans; when their values cover at most
// kStageBytes it first stages them in shared memory with coalesced loads. A lane then fits its own
// span when it is at most kLaneSpan long, tiles of eight lanes fit spans up to kTileSpan, the warp
// fits longer ones together, and spans longer than
// kWarpSpan (modes 2 and 3, not staged) go to the piece list, where many warps share their residual
// pass (k_pair_pieces, then k_pair_finish).
template <typename T, int MODE>
__global__ void __launch_bounds__(kGroupBlock, 3)
    k_span_groups(const T* __restrict__ v, const uint64_t* __restrict__ st, uint64_t count, uint32_t cap, int model,
                  const uint8_t* __restrict__ dirty, SpanStats* __restrict__ stats, uint64_t* __restrict__ size_out,
                  Record* __restrict__ rec, MergeWork mw) {
  constexpr int W = MODE == 2 ? 2 : 1;
  __shared__ __align__(16) unsigned char stage_raw[kGroupBlock / 32][kStageBytes];
  constexpr uint64_t kStageVals = kStageBytes / sizeof(T);
  const uint32_t lane = threadIdx.x & 31u, wib = threadIdx.x >> 5;
  T* stage = reinterpret_cast<T*>(stage_raw[wib]);
  const uint64_t ngroups = (count + 31) / 32;
  const uint64_t gw = (uint64_t)gridDim.x * (kGroupBlock / 32);
  for (uint64_t g = (uint64_t)blockIdx.x * (kGroupBlock / 32) + wib; g < ngroups; g += gw) {
    const uint64_t j = g * 32 + lane;
    bool act = j < count && (MODE != 2 || dirty[j]);
    if (!__any_sync(kFull, act)) continue;
    uint64_t a = 0, c = 0;
    if (act) {
      a = st[j];
      c = st[j + W];
      if (W == 2 && c - a > cap) {  // pairs beyond the cap never merge
        size_out[j] = kNone;
        act = false;
      }
    }
    const uint32_t N = act ? (uint32_t)(c - a) : 0u;
    const uint64_t ga = xw_min_u(act ? a : ~0ull), gc = xw_max_u(act ? c : 0ull);
    const bool staged = ga != ~0ull && gc - ga <= kStageVals;
    if (staged) {
      for (uint64_t t = lane; t < gc - ga; t += 32) stage[t] = __ldg(v + ga + t);
      __syncwarp();
    }
    const T* src = staged ? stage + (a - ga) : v + a;
    // moments
    SpanStats S;
    S.T0 = S.T1 = 0;
    S.mn = S.mx = 0;
    if (MODE == 1) {
      if (act && N <= kLaneSpan) S = stats_part(src, 0, N, 1);
      coop_stats<8>(__ballot_sync(kFull, act && N > kLaneSpan && N <= kTileSpan), src, N, S);
      coop_stats<32>(__ballot_sync(kFull, act && N > kTileSpan), src, N, S);
    } else if (MODE == 2 && act) {
      S = combine_stats(stats[j], st[j + 1] - a, stats[j + 1]);
    } else if (act) {
      S = stats[j];
    }
    // parameters (fit.cuh steps 1-3)
    const bool lin = model == LECO_MODEL_LINEAR && N >= 2;
    FitParams P;
    P.B = 0;
    P.fb_shift = 0;
    P.s = 0;
    P.fallback = 0;
    if (act) P = solve_params(lin ? 2 * S.T1 - mul_i128_u64(S.T0, N - 1) : (i128)0, S.mx, S.mn, N, lin);
    // residual range (step 4)
    int64_t lo = INT64_MAX, hi = INT64_MIN;
    uint64_t zmax = 0;
    const bool need = act && (lin || P.fallback);
    if (act && !need) {  // constant model on its grid: the residuals are the values
      lo = S.mn;
      hi = S.mx;
    }
    const bool by_lane = need && N <= kLaneSpan;
    const bool by_warp = need && N > kLaneSpan && (MODE == 1 || staged || N <= kWarpSpan);
    const bool by_pieces = need && !by_lane && !by_warp;
    if (by_lane) resid_part(src, 0, N, 1, P, lo, hi, zmax);
    coop_resid<8>(__ballot_sync(kFull, by_warp && N <= kTileSpan), src, N, P, lo, hi, zmax);
    coop_resid<32>(__ballot_sync(kFull, by_warp && N > kTileSpan), src, N, P, lo, hi, zmax);
    if (by_pieces) {
      const uint32_t np = (N + kPiece - 1) / kPiece;
      const unsigned long long li = atomicAdd(&mw.counters[0], 1ull);
      const unsigned long long pb = atomicAdd(&mw.counters[1], (unsigned long long)np);
      LongPair lp;
      lp.j = j;
      lp.k = 0;
      lp.a = a;
      lp.P = P;
      lp.N = N;
      lp.pad = 0;
      mw.longs[li] = lp;
      mw.lo[li] = INT64_MAX;
      mw.hi[li] = INT64_MIN;
      mw.zmax[li] = 0;
      for (uint32_t q = 0; q < np; q++) mw.pieces[pb + q] = ((uint64_t)li << 16) | q;
    }
    if (act && !by_pieces) {  // steps 5-6
      if (MODE == 3) {
        const FitResult R = finish_fit(P, lo, hi, zmax);
        Record r;
        r.theta0 = R.theta0;
        r.theta1 = R.theta1;
        r.start = a;
        r.word3 = make_w3(0, R.b, R.s, 1);
        rec[j] = r;
      } else {
        size_out[j] = kSmBits + (uint64_t)N * finish_width(P, lo, hi, zmax);
      }
      if (MODE == 1) stats[j] = S;
    }
    __syncwarp();  // the stage is reused by the next group
  }
}

// residual range of one piece of a long pair per warp, folded into the pair's range by atomics
template <typename T>
__global__ void __launch_bounds__(256) k_pair_pieces(const T* __restrict__ v, MergeWork mw) {
  const uint64_t np = *(volatile unsigned long long*)&mw.counters[1];
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nw = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  for (uint64_t pi = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; pi < np; pi += nw) {
    const uint64_t e = mw.pieces[pi];
    const uint64_t li = e >> 16;
    const uint32_t q = (uint32_t)(e & 0xFFFFu);
    const LongPair L = mw.longs[li];
    const uint32_t x0 = q * kPiece, x1 = min(x0 + kPiece, L.N);
    int64_t lo = INT64_MAX, hi = INT64_MIN;
    uint64_t z = 0;
    resid_part(v + L.a, x0 + lane, x1, 32, L.P, lo, hi, z);
    lo = warp_min_i64(lo);
    hi = warp_max_i64(hi);
    z = warp_max_u64(z);
    if (lane == 0) {
      atomicMin(&mw.lo[li], (long long)lo);
      atomicMax(&mw.hi[li], (long long)hi);
      atomicMax(&mw.zmax[li], (unsigned long long)z);
    }
  }
}

// steps 5-6 of the long spans: their merged size (msz) or their record (rec)
__global__ void k_pair_finish(MergeWork mw, uint64_t* __restrict__ msz, Record* __restrict__ rec) {
  const uint64_t nl = *(volatile unsigned long long*)&mw.counters[0];
  for (uint64_t li = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; li < nl; li += (uint64_t)gridDim.x * blockDim.x) {
    const LongPair L = mw.longs[li];
    if (rec) {
      const FitResult R = finish_fit(L.P, (int64_t)mw.lo[li], (int64_t)mw.hi[li], (uint64_t)mw.zmax[li]);
      Record r;
      r.theta0 = R.theta0;
      r.theta1 = R.theta1;
      r.start = L.a;
      r.word3 = make_w3(0, R.b, R.s, 1);
      rec[L.j] = r;
    } else {
      msz[L.j] = kSmBits + (uint64_t)L.N * finish_width(L.P, (int64_t)mw.lo[li], (int64_t)mw.hi[li], (uint64_t)mw.zmax[li]);
    }
  }
}

__device__ __forceinline__ bool pair_gain(const uint64_t* sz, const uint64_t* msz, uint64_t j, int64_t* g) {
  if (msz[j] == kNone) return false;
  *g = (int64_t)(sz[j] + sz[j + 1]) - (int64_t)msz[j];
  return true;
}

// priority order of two pairs: gain, then the hash of the start, then the smaller start
__device__ __forceinline__ bool beats(int64_t g1, uint64_t s1, int64_t g2, uint64_t s2) {
  if (g1 != g2) return g1 > g2;
  const uint64_t h1 = splitmix64(s1), h2 = splitmix64(s2);
  if (h1 != h2) return h1 > h2;
  return s1 < s2;
}

// sel[j]: pair j merges this round; keep[p]: partition p survives (it was not merged into its left
// neighbour); *nsel counts the merging pairs
__global__ void k_select(const uint64_t* __restrict__ st, const uint64_t* __restrict__ sz,
                         const uint64_t* __restrict__ msz, uint64_t m, uint8_t* __restrict__ sel,
                         uint64_t* __restrict__ keep, unsigned long long* __restrict__ nsel) {
  uint32_t local = 0;
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < m; j += (uint64_t)gridDim.x * blockDim.x) {
    bool ok = false;
    if (j + 1 < m) {
      int64_t g;
      ok = pair_gain(sz, msz, j, &g) && g > 0;
      if (ok && j > 0) {
        int64_t gl;
        if (pair_gain(sz, msz, j - 1, &gl) && !beats(g, st[j], gl, st[j - 1])) ok = false;
      }
      if (ok && j + 2 < m) {
        int64_t gr;
        if (pair_gain(sz, msz, j + 1, &gr) && !beats(g, st[j], gr, st[j + 1])) ok = false;
      }
    }
    sel[j] = ok ? 1 : 0;
    local += ok ? 1u : 0u;
    // partition j + 1 is absorbed when pair j merges; partition 0 always survives
    if (j + 1 < m) keep[j + 1] = ok ? 0ull : 1ull;
    if (j == 0) keep[0] = 1ull;
  }
  local = (uint32_t)warp_sum_u64(local);
  if ((threadIdx.x & 31u) == 0 && local) atomicAdd(nsel, (unsigned long long)local);
}

// the next round's arrays; a merged pair's moments are combined. Every load a partition needs is
// issued before the first branch, so the loads of one thread overlap.
__global__ void k_compact(const uint64_t* __restrict__ st, const uint64_t* __restrict__ sz,
                          const uint64_t* __restrict__ msz, const uint8_t* __restrict__ sel,
                          const uint64_t* __restrict__ newidx, const SpanStats* __restrict__ stats, uint64_t m,
                          uint64_t n, uint64_t new_m, uint64_t* __restrict__ nst, uint64_t* __restrict__ nsz,
                          uint64_t* __restrict__ nmsz, uint8_t* __restrict__ ndirty, SpanStats* __restrict__ nstats) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const bool absorbed = p > 0 && sel[p - 1];  // merged into p - 1
    const bool mp = p + 1 < m && sel[p];
    const bool mq2 = p + 3 < m && sel[p + 2];  // the next survivor's pair when p merges
    const bool mq1 = p + 2 < m && sel[p + 1];  // ... when it does not
    const uint64_t k = newidx[p];
    const uint64_t s0 = st[p];
    const uint64_t szp = sz[p];
    const uint64_t mszp = p + 1 < m ? msz[p] : 0;
    const uint64_t s1 = p + 1 < m ? st[p + 1] : n;
    if (absorbed) continue;
    const SpanStats sp = stats[p];
    nst[k] = s0;
    nsz[k] = mp ? mszp : szp;
    nstats[k] = mp ? combine_stats(sp, s1 - s0, stats[p + 1]) : sp;
    const uint64_t q = mp ? p + 2 : p + 1;  // next surviving partition
    if (q < m) {
      const bool d = mp || (mp ? mq2 : mq1);
      ndirty[k] = d ? 1 : 0;
      if (!d) nmsz[k] = mszp;
    }
    if (k == 0) nst[new_m] = n;
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

int group_grid(uint64_t count) {
  const uint64_t groups = (count + 31) / 32;
  return grid_for((groups + kGroupBlock / 32 - 1) / (kGroupBlock / 32), 1, 3);
}

// one mode of k_span_groups over count spans, then (modes 2 and 3) the pieces of the long ones
template <typename T>
cudaError_t span_groups(const void* values, int mode, const uint64_t* st, uint64_t count, uint32_t cap, int model,
                        const uint8_t* dirty, SpanStats* stats, uint64_t* size_out, Record* rec, const MergeWork& mw,
                        cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const T* v = static_cast<const T*>(values);
  if (mode != 1) {
    const cudaError_t e = cudaMemsetAsync(mw.counters, 0, 2 * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
  }
  if (mode == 1)
    k_span_groups<T, 1><<<group_grid(count), kGroupBlock, 0, s>>>(v, st, count, cap, model, dirty, stats, size_out,
                                                                  rec, mw);
  else if (mode == 2)
    k_span_groups<T, 2><<<group_grid(count), kGroupBlock, 0, s>>>(v, st, count, cap, model, dirty, stats, size_out,
                                                                  rec, mw);
  else
    k_span_groups<T, 3><<<group_grid(count), kGroupBlock, 0, s>>>(v, st, count, cap, model, dirty, stats, size_out,
                                                                  rec, mw);
  if (mode != 1) {
    k_pair_pieces<T><<<sm_count() * 8, 256, 0, s>>>(v, mw);
    k_pair_finish<<<sm_count() * 2, 256, 0, s>>>(mw, size_out, mode == 3 ? rec : nullptr);
  }
  return cudaGetLastError();
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

  // merge state
  const uint64_t m0 = m;
  SpanStats *stats = nullptr, *stats_b = nullptr;
  uint64_t *st_b = nullptr, *sz_a = nullptr, *sz_b = nullptr;
  uint64_t *msz_a = nullptr, *msz_b = nullptr, *keep = nullptr, *newidx = nullptr, *scr = nullptr, *d_total = nullptr;
  uint8_t *dirty_a = nullptr, *dirty_b = nullptr, *sel = nullptr;
  unsigned long long* d_nsel = nullptr;
  MergeWork mw;
  mw.longs = nullptr;
  mw.pieces = nullptr;
  mw.counters = nullptr;
  mw.lo = nullptr;
  mw.hi = nullptr;
  mw.zmax = nullptr;
  const uint64_t long_cap = 2 * n / kWarpSpan + 2;
  const uint64_t piece_cap = 2 * n / kPiece + long_cap + 2;
  const uint64_t scr_elems = m0 / 2048 + 2;
  if (e == cudaSuccess) e = dalloc(&stats, m0, st);
  if (e == cudaSuccess) e = dalloc(&stats_b, m0, st);
  if (e == cudaSuccess) e = dalloc(&st_b, m0 + 1, st);
  if (e == cudaSuccess) e = dalloc(&sz_a, m0, st);
  if (e == cudaSuccess) e = dalloc(&sz_b, m0, st);
  if (e == cudaSuccess) e = dalloc(&msz_a, m0, st);
  if (e == cudaSuccess) e = dalloc(&msz_b, m0, st);
  if (e == cudaSuccess) e = dalloc(&keep, m0, st);
  if (e == cudaSuccess) e = dalloc(&newidx, m0, st);
  if (e == cudaSuccess) e = dalloc(&scr, scr_elems + 1, st);
  if (e == cudaSuccess) e = dalloc(&d_total, 1, st);
  if (e == cudaSuccess) e = dalloc(&dirty_a, m0, st);
  if (e == cudaSuccess) e = dalloc(&dirty_b, m0, st);
  if (e == cudaSuccess) e = dalloc(&sel, m0, st);
  if (e == cudaSuccess) e = dalloc(&d_nsel, 1, st);
  if (e == cudaSuccess) e = dalloc(&mw.longs, long_cap, st);
  if (e == cudaSuccess) e = dalloc(&mw.pieces, piece_cap, st);
  if (e == cudaSuccess) e = dalloc(&mw.counters, 2, st);
  if (e == cudaSuccess) e = dalloc(&mw.lo, long_cap, st);
  if (e == cudaSuccess) e = dalloc(&mw.hi, long_cap, st);
  if (e == cudaSuccess) e = dalloc(&mw.zmax, long_cap, st);
  uint64_t* cur_st = starts_out;
  uint64_t* nxt_st = st_b;
  // every split partition's moments, fit and size
  if (e == cudaSuccess)
    e = u32 ? span_groups<uint32_t>(values, 1, cur_st, m, cap, model, nullptr, stats, sz_a, nullptr, mw, st)
            : span_groups<uint64_t>(values, 1, cur_st, m, cap, model, nullptr, stats, sz_a, nullptr, mw, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(dirty_a, 1, m, st);
  while (e == cudaSuccess && m > 1) {
    e = u32 ? span_groups<uint32_t>(values, 2, cur_st, m - 1, cap, model, dirty_a, stats, msz_a, nullptr, mw, st)
            : span_groups<uint64_t>(values, 2, cur_st, m - 1, cap, model, dirty_a, stats, msz_a, nullptr, mw, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_nsel, 0, 8, st);
    if (e != cudaSuccess) break;
    k_select<<<grid_for(m, 256, 8), 256, 0, st>>>(cur_st, sz_a, msz_a, m, sel, keep, d_nsel);
    unsigned long long nsel = 0;
    e = cudaMemcpyAsync(&nsel, d_nsel, 8, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess || nsel == 0) break;
    e = scan_u64(keep, m, newidx, scr, d_total, st);
    if (e != cudaSuccess) break;
    const uint64_t new_m = m - nsel;
    k_compact<<<grid_for(m, 256, 8), 256, 0, st>>>(cur_st, sz_a, msz_a, sel, newidx, stats, m, n, new_m, nxt_st,
                                                   sz_b, msz_b, dirty_b, stats_b);
    e = cudaGetLastError();
    std::swap(cur_st, nxt_st);
    std::swap(sz_a, sz_b);
    std::swap(msz_a, msz_b);
    std::swap(dirty_a, dirty_b);
    std::swap(stats, stats_b);
    m = new_m;
  }
  if (e == cudaSuccess && rec_out) {
    e = dalloc(rec_out, m, st);  // the final partitions' fits from their moments
    if (e == cudaSuccess)
      e = u32 ? span_groups<uint32_t>(values, 3, cur_st, m, cap, model, nullptr, stats, nullptr, *rec_out, mw, st)
              : span_groups<uint64_t>(values, 3, cur_st, m, cap, model, nullptr, stats, nullptr, *rec_out, mw, st);
  }
  if (e == cudaSuccess && cur_st != starts_out)
    e = cudaMemcpyAsync(starts_out, cur_st, (m + 1) * 8, cudaMemcpyDeviceToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFreeAsync(cur_st == starts_out ? nxt_st : cur_st, st);  // st_b, wherever it ended up
  for (void* p : {(void*)stats, (void*)stats_b, (void*)sz_a,
                  (void*)sz_b, (void*)msz_a, (void*)msz_b, (void*)keep, (void*)newidx, (void*)scr, (void*)d_total,
                  (void*)dirty_a, (void*)dirty_b, (void*)sel, (void*)d_nsel, (void*)mw.longs, (void*)mw.pieces,
                  (void*)mw.counters, (void*)mw.lo, (void*)mw.hi, (void*)mw.zmax})
    if (p) cudaFreeAsync(p, st);
  if (e != cudaSuccess && rec_out && *rec_out) {
    cudaFreeAsync(*rec_out, st);
    *rec_out = nullptr;
  }
  if (e == cudaSuccess) *m_out = m;
  return e;
}

cudaError_t var_partition(const void* values, int dtype, uint64_t n, double tau, uint32_t cap, int model, bool seeded,
                          uint64_t* starts_out, uint64_t* m_out, cudaStream_t st) {
  return var_partition_fit(values, dtype, n, tau, cap, model, seeded, starts_out, m_out, nullptr, st);
}

cudaError_t var_partition(const void* values, int dtype, uint64_t n, double tau, uint32_t cap,
                          int model, uint64_t* starts_out, uint64_t* m_out, cudaStream_t st) {
  return var_partition_fit(values, dtype, n, tau, cap, model, false, starts_out, m_out, nullptr, st);
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

