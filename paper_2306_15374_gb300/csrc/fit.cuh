// Partition fit shared by the encoder and the variable-length partitioner (§3.1 Regressor).
//
// Fit of one partition of N values (w = the value as two's complement int64):
//  1. exact least-squares slope q = 6S/D, S = sum (2x - (N-1)) (w_x - w_0), D = N (N^2 - 1)
//     (integer moments reduced across the group in int128; q = 0 for the constant model; the
//     quotients are exact, by the reciprocal of D, see solve_params);
//  2. magnitude bound U = max|w| + (wmax - wmin) + (ceil|q| + 1) N + 4; bitlen(U) > 62 falls back
//     to the constant model on the grid 2^11 (residuals taken mod 2^64);
//  3. grid exponent s = min(52, 52 - bitlen(U)), slope B = round(q 2^s) (half up);
//  4. residual range [lo, hi] of r0_x = w_x - floor(B x 2^-s) (a second pass);
//  5. minimax intercept t = lo + ceil((hi - lo)/2), rounded down to the grid step 2^max(0,-s);
//  6. width b = bitlen(max(zigzag(lo - t), zigzag(hi - t))) (zigzag is V-shaped, so the extremes
//     of the residual range carry the maximum).
// The bound makes theta0 = A 2^-s and theta1 = B 2^-s exact binary64 numbers whose prediction
// floor(fl(fl(theta1 x) + theta0)) equals the integer (A + B x) >> s for every x < N.
#pragma once

#include "leco_internal.cuh"

namespace leco {
namespace {

// (u1 2^64 + u0) / v for u1 < v (so the quotient fits 64 bits), with the remainder: schoolbook
// long division in base 2^32 after normalising v (Knuth's algorithm D with two quotient digits, in
// the form of Warren's "divlu", Hacker's Delight §9-4). Each digit is estimated from the top two
// dividend digits over the top divisor digit and corrected at most twice.
__device__ __forceinline__ uint64_t divlu(uint64_t u1, uint64_t u0, uint64_t v, uint64_t* rem) {
  const uint64_t base = 1ull << 32;
  const int sh = __clzll((long long)v);  // v > 0
  v <<= sh;
  const uint64_t vn1 = v >> 32, vn0 = v & 0xFFFFFFFFull;
  const uint64_t un32 = sh ? (u1 << sh) | (u0 >> (64 - sh)) : u1;
  const uint64_t un10 = u0 << sh;
  const uint64_t un1 = un10 >> 32, un0 = un10 & 0xFFFFFFFFull;
  uint64_t q1 = un32 / vn1, rhat = un32 - q1 * vn1;
  while (q1 >= base || q1 * vn0 > base * rhat + un1) {
    q1--;
    rhat += vn1;
    if (rhat >= base) break;
  }
  const uint64_t un21 = un32 * base + un1 - q1 * v;
  uint64_t q0 = un21 / vn1;
  rhat = un21 - q0 * vn1;
  while (q0 >= base || q0 * vn0 > base * rhat + un0) {
    q0--;
    rhat += vn1;
    if (rhat >= base) break;
  }
  *rem = (un21 * base + un0 - q0 * v) >> sh;
  return q1 * base + q0;
}

// floor(num / den) for den > 0, exactly: what the reciprocals below do not serve (grids coarser than 1,
// partitions beyond 2^21 values, the Gram norms). Divisors below 2^64 take one native 64-bit division when
// |num| < 2^64, else two native 64-bit divisions and one 128-by-64 long division; wider divisors use the generic
// 128-bit routine, whose bit-serial latency would otherwise stall a whole CTA per fitted partition.
__device__ __forceinline__ i128 floordiv_i128(i128 num, i128 den) {
  if ((den >> 64) == 0 && num != ((i128)1 << 127)) {
    const uint64_t d = (uint64_t)den;
    const bool neg = num < 0;
    const u128 u = neg ? (u128)0 - (u128)num : (u128)num;
    const uint64_t hi = (uint64_t)(u >> 64), lo = (uint64_t)u;
    if (hi == 0) {
      const uint64_t q0 = lo / d, r0 = lo - q0 * d;
      return neg ? -(i128)q0 - (r0 != 0 ? 1 : 0) : (i128)q0;
    }
    const uint64_t qh = hi / d;
    uint64_t r = 0;
    const uint64_t ql = divlu(hi - qh * d, lo, d, &r);
    const u128 q = ((u128)qh << 64) | ql;
    return neg ? -(i128)q - (r != 0 ? 1 : 0) : (i128)q;
  }
  i128 t = num / den;
  if ((num % den) != 0 && num < 0) t -= 1;
  return t;
}

__device__ __forceinline__ i128 round_half_up_i128(i128 num, i128 den) {  // den > 0
  return floordiv_i128(2 * num + den, 2 * den);
}

__device__ __forceinline__ double pow2(int e) {  // exact 2^e for -1022 <= e <= 1023
  return __longlong_as_double((long long)(1023 + e) << 52);
}

struct FitParams {
  int64_t B;
  int64_t fb_shift;  // fallback: theta0 as an integer (multiple of 2^11)
  int32_t s;
  int16_t fallback;
  int16_t narrow;    // fit_range: the second pass fits 32 bits
};

struct FitResult {
  double theta0;
  double theta1;
  int32_t s;
  uint32_t b;
};

// Reciprocals of the least-squares denominators D(N) = N (N^2 - 1): v = floor((2^128 - 1) / d) - 2^64
// for the divisor d = D normalised (shifted left until its top bit is set), as in Moeller & Granlund,
// "Improved division by invariant integers" (IEEE Trans. Computers 60(2), 2011). D depends on the
// partition length alone, so the table (32 KB, short lengths in L1) turns every division of the
// solve into a high product and two corrections; longer partitions compute v once per solve.
constexpr uint32_t kRecipLen = 4096;

struct RecipTable {
  uint64_t v[kRecipLen + 1];
};

constexpr RecipTable make_recip_table() {
  RecipTable t{};
  for (uint64_t N = 2; N <= kRecipLen; N++) {
    uint64_t d = N * (N * N - 1);
    while (!(d >> 63)) d <<= 1;
    t.v[N] = (uint64_t)(~(u128)0 / d);  // the quotient lies in [2^64, 2^65): its low word
  }
  return t;
}

static __device__ const RecipTable kRecip = make_recip_table();

__device__ __forceinline__ int clz64(uint64_t x) { return __clzll((long long)x); }  // x > 0

// floor((u1 2^64 + u0) / d) for a normalised d with reciprocal v and u1 < d (Moeller & Granlund,
// algorithm 4)
__device__ __forceinline__ uint64_t div_recip(uint64_t u1, uint64_t u0, uint64_t d, uint64_t v) {
  uint64_t q0 = v * u1, q1 = __umul64hi(v, u1);
  q0 += u0;
  q1 += u1 + (q0 < u0 ? 1ull : 0ull) + 1ull;
  uint64_t r = u0 - q1 * d;
  if (r > q0) {
    q1--;
    r += d;
  }
  return r >= d ? q1 + 1 : q1;
}

__device__ __forceinline__ uint64_t recip_of(uint64_t dn) {  // as the table's entries
  uint64_t rem;
  return divlu(~dn, ~0ull, dn, &rem);  // (2^128 - 1) - 2^64 dn over dn
}

// the constant model on the grid 2^11, for partitions whose magnitude bound exceeds 62 bits (step 2)
__device__ __forceinline__ FitParams fallback_params(int64_t mx, int64_t mn) {
  const uint64_t half = (uint64_t)mx - (uint64_t)mn;  // mx - mn < 2^64
  // mn + ceil((mx - mn) / 2) rounded down to a multiple of 2^11
  const int64_t t = (int64_t)((uint64_t)mn + (half >> 1) + (half & 1ull));
  FitParams P;
  P.fallback = 1;
  P.s = -11;
  P.B = 0;
  P.fb_shift = (t >> 11) * 2048;
  P.narrow = 0;
  return P;
}

constexpr uint32_t kFastLen = 1u << 21;  // D(N) < 2^63: the divisions below take one 64-bit divisor

// The usual line, branch-free: 2 <= N <= kRecipLen, |S| < 2^58 and |values| < 2^62, so that the first
// dividend and the magnitude bound are plain words. False when the grid is coarser than 1 (s < 0), which
// also holds whenever the bound asks for the fallback; solve_params then takes the general way. The merge
// rounds solve a line per pair: 100M piecewise values 18.95 -> 18.6 ms, k_fit_spans 7.25 -> 7.0 ms.
__device__ __forceinline__ bool solve_short(int64_t S, int64_t mx, int64_t mn, uint32_t N, FitParams* P) {
  const uint64_t amx = (uint64_t)(mx < 0 ? -mx : mx), amn = (uint64_t)(mn < 0 ? -mn : mn);
  const uint64_t base = (amx > amn ? amx : amn) + ((uint64_t)mx - (uint64_t)mn) + 4;
  const bool neg = S < 0;
  const uint64_t a6 = (uint64_t)(neg ? -S : S) * 6;
  const uint64_t d = (uint64_t)N * (N * N - 1);
  const int sh = clz64(d);  // 28 .. 61
  const uint64_t dn = d << sh;
  const uint64_t v = kRecip.v[N];
  const uint64_t t = a6 + (d - 1);
  const uint64_t Q = div_recip(t >> (64 - sh), t << sh, dn, v);
  const int s = clz64(base + (Q + 1) * N) - 12;
  if (s < 0) return false;
  // (2 |6S| 2^s + D or D - 1) / 2D, both sides normalised
  const int k = s + sh;
  const uint64_t add = (d - (neg ? 1u : 0u)) << (sh - 1);
  const uint64_t l0 = k < 64 ? a6 << k : 0, h0 = k < 64 ? a6 >> (64 - k) : a6 << (k - 64);
  const uint64_t lo = l0 + add;
  const uint64_t q = div_recip(h0 + (lo < l0 ? 1u : 0u), lo, dn, v);
  P->fallback = 0;
  P->s = s;
  P->B = neg ? -(int64_t)q : (int64_t)q;
  P->fb_shift = 0;
  P->narrow = 0;
  return true;
}

// step 1-3 (one thread): parameters from the reduced moments. Each of the two quotients, ceil(|q|) for
// the magnitude bound and round(q 2^s), is below 2^64 whenever it is used, so it takes one
// 128-by-64-bit step by the reciprocal of D; a quotient that would not fit puts the bound above
// 62 bits. Against three 64-bit divisions and 128-bit bounds: partition + encode of 100M piecewise
// values 35.15 -> 34.50 ms, of 250M 32-bit timestamps 19.82 -> 19.60 ms.
__device__ FitParams solve_params(i128 S, int64_t mx, int64_t mn, uint32_t N, bool lin) {
  const int64_t lim = (int64_t)1 << 62;
  if (lin && N >= 2 && N <= kRecipLen && S > -((i128)1 << 58) && S < ((i128)1 << 58) && mx < lim && mn > -lim) {
    FitParams P;
    if (solve_short((int64_t)S, mx, mn, N, &P)) return P;
  }
  // U > max|w| and U > mx - mn: bits above 62 there decide the fallback
  if (mx >= lim || mn <= -lim || (uint64_t)mx - (uint64_t)mn >= (uint64_t)lim) return fallback_params(mx, mn);
  const uint64_t amx = (uint64_t)(mx < 0 ? -mx : mx), amn = (uint64_t)(mn < 0 ? -mn : mn);
  const uint64_t base = (amx > amn ? amx : amn) + ((uint64_t)mx - (uint64_t)mn) + 4;  // < 2^63 + 4
  const bool neg = S < 0;
  uint64_t Q = 0;
  i128 D = 1;
  uint64_t dn = 0, v = 0;
  int sh = 0;
  u128 a6 = 0;
  const bool fast = N <= kFastLen;
  if (lin) {
    const u128 aS = neg ? (u128)0 - (u128)S : (u128)S;
    a6 = aS * 6;  // |S| <= 2^62 N^2 < 2^110
    if (N == 2) {
      if (aS >> 62) return fallback_params(mx, mn);
      Q = (uint64_t)aS;  // D = 6
    } else if (fast) {
      const uint64_t d = (uint64_t)N * ((uint64_t)N * N - 1);
      D = (i128)d;
      sh = clz64(d);  // >= 1
      dn = d << sh;
      v = N <= kRecipLen ? kRecip.v[N] : recip_of(dn);
      const u128 t = a6 + (d - 1);
      if ((uint64_t)(t >> 64) == 0) {
        Q = div_recip((uint64_t)t >> (64 - sh), (uint64_t)t << sh, dn, v);
      } else {
        if (t >> (128 - sh)) return fallback_params(mx, mn);  // the quotient exceeds 64 bits
        const u128 tn = t << sh;
        if ((uint64_t)(tn >> 64) >= dn) return fallback_params(mx, mn);
        Q = div_recip((uint64_t)(tn >> 64), (uint64_t)tn, dn, v);
      }
    } else {
      D = (i128)((u128)(uint64_t)N * ((uint64_t)N * N - 1));
      const i128 q = floordiv_i128((i128)a6 + D - 1, D);
      if (q >> 62) return fallback_params(mx, mn);
      Q = (uint64_t)q;
    }
    if (Q >> 62) return fallback_params(mx, mn);
  }
  // U = base + (Q + 1) N
  if (__umul64hi(Q + 1, N)) return fallback_params(mx, mn);
  const uint64_t g = (Q + 1) * N;
  if ((g >> 62) || ((base + g) >> 62)) return fallback_params(mx, mn);
  const int eU = 64 - clz64(base + g);  // base >= 4
  const int s = 52 - eU;                  // -10 .. 49
  int64_t B = 0;
  if (lin && N == 2) {  // q = S exactly: B = S 2^s, or round(S / 2^-s) half up by a shift
    const int64_t q = (int64_t)S;
    B = s >= 0 ? (int64_t)((uint64_t)q << s) : (2 * q + ((int64_t)1 << (-s))) >> (1 - s);
  } else if (lin && fast && s >= 0) {
    // floor((2 a + D) / 2D) for q >= 0, -floor((2 a + D - 1) / 2D) below 0, with a = |6S| 2^s; the
    // result is below 2^53, so the dividend's high word is below the divisor's
    // (2D normalised is D normalised: one place less)
    uint64_t q;
    if ((uint64_t)(a6 >> 64) == 0 && ((uint64_t)a6 >> (62 - s)) == 0) {
      const uint64_t t = ((uint64_t)a6 << (s + 1)) + (uint64_t)D - (neg ? 1u : 0u);  // D < 2^63
      q = div_recip((t >> 1) >> (64 - sh), t << (sh - 1), dn, v);
    } else {
      const u128 t = ((a6 << s) << 1) + (u128)D - (neg ? 1u : 0u);
      const u128 tn = t << (sh - 1);
      q = div_recip((uint64_t)(tn >> 64), (uint64_t)tn, dn, v);
    }
    B = neg ? -(int64_t)q : (int64_t)q;
  } else if (lin) {
    const i128 sixS = neg ? -(i128)a6 : (i128)a6;
    B = (int64_t)(s >= 0 ? round_half_up_i128((i128)((u128)sixS << s), D)
                         : round_half_up_i128(sixS, (i128)((u128)D << (-s))));
  }
  FitParams P;
  P.fallback = 0;
  P.s = s;
  P.B = B;
  P.fb_shift = 0;
  P.narrow = 0;
  return P;
}

// step 6 alone (one thread): the width b, without the binary64 parameters (sizing only)
__device__ __forceinline__ uint32_t finish_width(const FitParams& P, int64_t lo, int64_t hi, uint64_t fb_maxzz) {
  if (P.fallback) return (uint32_t)bitlen_u64(fb_maxzz);
  const int s = P.s;
  // without a grid the intercept centres the range exactly: the wider zigzag code is hi - lo itself
  // (2k - 1 and 2k for an even range 2k, 2k + 1 and 2k for an odd one)
  if (s >= 0) return (uint32_t)bitlen_u64((uint64_t)hi - (uint64_t)lo);
  const i128 t = (i128)lo + (((i128)hi - (i128)lo + 1) >> 1);
  const i128 shift = (t >> (-s)) * ((i128)1 << (-s));
  const int64_t lo2 = (int64_t)((i128)lo - shift), hi2 = (int64_t)((i128)hi - shift);
  return (uint32_t)bitlen_u64(max(zz_encode(lo2), zz_encode(hi2)));
}

// steps 5-6 (one thread)
__device__ FitResult finish_fit(const FitParams& P, int64_t lo, int64_t hi, uint64_t fb_maxzz) {
  FitResult R;
  if (P.fallback) {
    R.theta0 = (double)P.fb_shift;  // multiple of 2^11 with |.| <= 2^63: exact
    R.theta1 = 0.0;
    R.s = -11;
    R.b = (uint32_t)bitlen_u64(fb_maxzz);
    return R;
  }
  const int s = P.s;
  // the residuals lie in (-2^62, 2^62) (step 2), so their midpoint and range fit 64 bits
  const uint64_t d = (uint64_t)hi - (uint64_t)lo;
  const int64_t t = lo + (int64_t)((d >> 1) + (d & 1ull));
  const int64_t A = s >= 0 ? (int64_t)((uint64_t)t << s) : t >> (-s);  // |A| < 2^53
  R.b = finish_width(P, lo, hi, 0);
  R.s = s;
  R.theta0 = (double)A * pow2(-s);
  R.theta1 = (double)P.B * pow2(-s);
  return R;
}


// Narrow spans: values within 2^30 of a reference in (-2^62, 2^62), so that their differences d from it fit
// 32 bits (a difference that wraps in 64 bits is above 2^61 in magnitude, so the test sees it), and a line
// that stays within 2^30 over the span. Extremes are then 32-bit, products 32 x 32 -> 64-bit, and the line
// needs no 64-bit shift: G = B x 2^(32-s) (or B x, for s > 32) is carried and its high half read.
constexpr int64_t kNarrow = (int64_t)1 << 30;
constexpr int64_t kNarrowRef = (int64_t)1 << 62;
__device__ __forceinline__ bool narrow_ref(int64_t ref) { return ref > -kNarrowRef && ref < kNarrowRef; }
__device__ __forceinline__ bool narrow_diff(int64_t d) { return d > -kNarrow && d < kNarrow; }
__device__ __forceinline__ bool narrow_line(const FitParams& P, uint32_t N) {
  return !P.fallback && P.s >= 0 && ((uint64_t)(P.B < 0 ? -P.B : P.B) * (N - 1)) >> P.s < (uint64_t)kNarrow;
}
struct NarrowLine {
  uint64_t B;
  uint32_t sh;
  __device__ __forceinline__ NarrowLine(int64_t slope, int s)
      : B((uint64_t)slope << (s < 32 ? 32 - s : 0)), sh(s > 32 ? (uint32_t)(s - 32) : 0u) {}
  __device__ __forceinline__ int32_t at(uint64_t G) const { return (int32_t)(G >> 32) >> sh; }
};

// Group fit: GROUP threads (one thread, a warp, or a whole CTA when GROUP > 32) fit [a, a+N).
// Returns the result in every thread of the group. sm: shared scratch (only used when GROUP > 32).
struct FitShared {
  i128 S[32];
  int64_t mx[32], mn[32];
  uint64_t zmax[32];
  FitParams P;
  FitResult R;
};

// f over one group member's values v[rank], v[rank + GROUP], ... of N, RUN at a time with their loads in
// flight together (whole runs without bounds; the last one repeats v[0] past the end); stops when f's run
// hook `ok` says so
template <int GROUP, int RUN, typename T, typename F, typename Ok>
__device__ __forceinline__ bool for_runs(const T* __restrict__ v, uint32_t N, uint32_t rank, T ref, F f, Ok ok) {
  const T* p = v + rank;
  // whole runs are the same for all members: the values of one run of the group lie side by side
  uint32_t left = N;
  for (; left >= (uint32_t)(RUN * GROUP); left -= RUN * GROUP, p += RUN * GROUP) {
    T w[RUN];
#pragma unroll
    for (int k = 0; k < RUN; k++) w[k] = __ldg(p + k * GROUP);
#pragma unroll
    for (int k = 0; k < RUN; k++) f(w[k]);
    if (!ok()) return false;
  }
  if (left) {
    const int mine = left > rank ? (int)((left - rank - 1) / GROUP) + 1 : 0;
    T w[RUN];
#pragma unroll
    for (int k = 0; k < RUN; k++) w[k] = k < mine ? __ldg(p + k * GROUP) : ref;
#pragma unroll
    for (int k = 0; k < RUN; k++)
      if (k < mine) f(w[k]);
    if (!ok()) return false;
  }
  return true;
}

// Pass 1 over one group member's positions x = rank, rank + GROUP, ... < N of the values v (the
// partition's first value at v[0]): min, max and (linear model) S = sum u_x w_x with
// u_x = 2x - (N-1), where w is the value as two's complement int64 (over the whole group S equals
// sum u_x (w_x - w_0) because the u_x sum to zero). Narrow partitions take their differences from w_0 in
// 32 bits; a group that meets a value too far away starts again in 64 bits: each term is then split as
// u w_hi 2^32 + u w_lo with 32 x 32 -> 64-bit products, accumulated in 64 bits over at most 64 terms
// (|u| < 2^24: each partial stays below 2^62) and folded into 128 bits. Pairs of warps on one partition
// (GROUP 64, partitions of 1024+ values) keep sixteen loads in flight per lane, warps eight.
// In 64 bits throughout, with bounds on every load, the two passes took 43 instructions per value and
// were bound by their issue: 200M sorted normal uint64 in partitions of 4096 414 -> 307 us (1.6 GB read),
// 20M 32-bit values in partitions of 1000 51 -> 32 us, 96 columns of 200M values 600 -> 490 us.
struct NarrowMom {
  int64_t S;        // sum of u_x (w_x - w_0) over the member's positions
  int32_t mx, mn;   // of w_x - w_0; w_0 itself counts
};

template <int GROUP, typename T>
__device__ __forceinline__ bool fit_pass1_narrow(const T* __restrict__ v, uint32_t N, bool lin, uint32_t rank, int64_t ref,
                                                 NarrowMom& out) {
  if (!narrow_ref(ref) || N > (1u << 16)) return false;  // |u| < 2^16, 2^30 differences, 2^11 values: below 2^57
  int32_t mx = 0, mn = 0;
  int32_t u = 2 * (int32_t)rank - ((int32_t)N - 1);
  uint32_t far = 0;
  int64_t S = 0;
  auto add = [&](T value) {
    const int64_t d = (int64_t)value - ref;
    const int32_t e = (int32_t)d;
    far |= (uint32_t)((int32_t)(d >> 32) ^ (e >> 31));  // d outside 32 bits
    mx = max(mx, e);
    mn = min(mn, e);
    if (lin) S += (int64_t)u * e;
    u += 2 * GROUP;
  };
  auto ok = [&]() { return !__any_sync(0xffffffffu, far != 0 || mn <= -(int32_t)kNarrow || mx >= (int32_t)kNarrow); };
  if (!for_runs<GROUP, GROUP == 64 ? 16 : 8>(v, N, rank, (T)ref, add, ok)) return false;
  out.S = S;
  out.mx = mx;
  out.mn = mn;
  return true;
}

// pass 2 of a narrow partition: the member's residual range, relative to w_0 (empty members: the inverted range)
template <int GROUP, typename T>
__device__ __forceinline__ void fit_pass2_narrow(const T* __restrict__ v, uint32_t N, int64_t B, int32_t s, uint32_t rank,
                                                 int64_t ref, int32_t* lo, int32_t* hi) {
  const NarrowLine line(B, s);
  int32_t l = INT32_MAX, h = INT32_MIN;
  uint64_t G = line.B * rank;
  const uint64_t dG = line.B * (uint64_t)GROUP;
  const uint32_t r32 = (uint32_t)ref;
  auto add = [&](T value) {
    const int32_t r = (int32_t)((uint32_t)value - r32) - line.at(G);
    l = min(l, r);
    h = max(h, r);
    G += dG;
  };
  for_runs<GROUP, GROUP == 64 ? 16 : 8>(v, N, rank, (T)ref, add, []() { return true; });
  *lo = l;
  *hi = h;
}

template <int GROUP, typename T>
__device__ __forceinline__ void fit_pass1_wide(const T* __restrict__ v, uint32_t N, bool lin, uint32_t rank, i128* S_out,
                                               int64_t* mx_out, int64_t* mn_out) {
  int64_t mx = INT64_MIN, mn = INT64_MAX;
  i128 S = 0;
  if (lin) {
    const int64_t nm1 = (int64_t)N - 1;
    for (uint32_t x0 = rank; x0 < N; x0 += 64u * GROUP) {
      const uint32_t xe = N - x0 > 64u * GROUP ? x0 + 64u * GROUP : N;
      int64_t acc_hi = 0, acc_lo = 0;
      int32_t u = (int32_t)(2 * (int64_t)x0 - nm1);
#pragma unroll 8
      for (uint32_t x = x0; x < xe; x += GROUP, u += 2 * GROUP) {
        const int64_t w = (int64_t)__ldg(v + x);
        mx = max(mx, w);
        mn = min(mn, w);
        if (sizeof(T) == 8) acc_hi += (int64_t)u * (int64_t)(int32_t)(w >> 32);
        acc_lo += (int64_t)u * (int64_t)(uint32_t)w;
      }
      S += (i128)acc_hi * ((i128)1 << 32) + (i128)acc_lo;
    }
  } else {
#pragma unroll 8
    for (uint32_t x = rank; x < N; x += GROUP) {
      const int64_t w = (int64_t)__ldg(v + x);
      mx = max(mx, w);
      mn = min(mn, w);
    }
  }
  *S_out = S;
  *mx_out = mx;
  *mn_out = mn;
}

template <int GROUP, typename T>
__device__ __forceinline__ void fit_pass1(const T* __restrict__ v, uint32_t N, bool lin, uint32_t rank, i128* S_out,
                                          int64_t* mx_out, int64_t* mn_out) {
  NarrowMom m;
  if (GROUP > 1) {
    const int64_t ref = (int64_t)__ldg(v);
    if (fit_pass1_narrow<GROUP>(v, N, lin, rank, ref, m)) {
      // as a sum of u w: the member's u add up to cnt (2 rank - (N-1)) + GROUP cnt (cnt - 1)
      const int64_t cnt = rank < N ? (int64_t)((N - 1 - rank) / GROUP + 1) : 0;
      *S_out = lin ? (i128)m.S + mul_s64(ref, cnt * (2 * (int64_t)rank - ((int64_t)N - 1)) + (int64_t)GROUP * cnt * (cnt - 1))
                   : (i128)0;
      *mx_out = ref + m.mx;
      *mn_out = ref + m.mn;
      return;
    }
  }
  fit_pass1_wide<GROUP>(v, N, lin, rank, S_out, mx_out, mn_out);
}

// Pass 2: range [lo, hi] of the residuals w_x - line(x) with line(x) = (B x) >> s (s >= 0) or
// (B x) << -s, B x taken mod 2^64 and stepped by B GROUP from one position to the next; in 32 bits
// when the partition and its line are narrow.
template <int GROUP, typename T>
__device__ __forceinline__ void fit_pass2(const T* __restrict__ v, uint32_t N, const FitParams& P, uint32_t rank,
                                          int64_t* lo_out, int64_t* hi_out) {
  if (GROUP > 1 && P.narrow) {
    const int64_t ref = (int64_t)__ldg(v);
    int32_t l, h;
    fit_pass2_narrow<GROUP>(v, N, P.B, P.s, rank, ref, &l, &h);
    *lo_out = rank < N ? ref + l : INT64_MAX;
    *hi_out = rank < N ? ref + h : INT64_MIN;
    return;
  }
  const int64_t B = P.B;
  const int32_t s = P.s;
  int64_t lo = INT64_MAX, hi = INT64_MIN;
  uint64_t F = (uint64_t)B * rank;
  const uint64_t dF = (uint64_t)B * GROUP;
  if (s >= 0) {
#pragma unroll 8
    for (uint32_t x = rank; x < N; x += GROUP, F += dF) {
      const int64_t r = (int64_t)__ldg(v + x) - ((int64_t)F >> s);
      lo = min(lo, r);
      hi = max(hi, r);
    }
  } else {
    for (uint32_t x = rank; x < N; x += GROUP, F += dF) {
      const int64_t r = (int64_t)__ldg(v + x) - (int64_t)(F << (-s));
      lo = min(lo, r);
      hi = max(hi, r);
    }
  }
  *lo_out = lo;
  *hi_out = hi;
}

// barrier of a fitting group wider than a warp: the CTA (bar_id < 0) or named barrier bar_id over
// the group's nthreads threads (several groups in one CTA)
__device__ __forceinline__ void group_sync(int bar_id, uint32_t nthreads) {
  if (bar_id < 0)
    __syncthreads();
  else
    asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(nthreads) : "memory");
}

template <int GROUP>
__device__ FitResult fit_range(const void* __restrict__ values, int dtype, uint64_t a, uint32_t N,
                               int model, uint32_t rank, FitShared* sm, int bar_id = -1) {
  const bool lin = model == LECO_MODEL_LINEAR && N >= 2;
  const bool u32 = dtype == LECO_U32;
  const uint32_t* v32 = static_cast<const uint32_t*>(values) + a;
  const uint64_t* v64 = static_cast<const uint64_t*>(values) + a;
  i128 S;
  int64_t mx, mn;
  if (u32)
    fit_pass1<GROUP>(v32, N, lin, rank, &S, &mx, &mn);
  else
    fit_pass1<GROUP>(v64, N, lin, rank, &S, &mx, &mn);
  if (GROUP > 1) {
    S = warp_sum_i128(S);
    mx = warp_max_i64(mx);
    mn = warp_min_i64(mn);
  }
  const uint32_t lane = rank & 31u;
  FitParams P;
  auto solve = [&](i128 moment) {
    FitParams q = solve_params(moment, mx, mn, N, lin);
    q.narrow = narrow_line(q, N) && narrow_ref(mn) && narrow_diff(mx - mn) ? 1 : 0;
    return q;
  };
  if (GROUP == 1) {
    P = solve(S);
  } else if (GROUP == 32) {
    if (lane == 0) P = solve(S);
    P.B = (int64_t)__shfl_sync(0xffffffffu, (unsigned long long)P.B, 0);
    P.fb_shift = (int64_t)__shfl_sync(0xffffffffu, (unsigned long long)P.fb_shift, 0);
    P.s = __shfl_sync(0xffffffffu, P.s, 0);
    const uint32_t f = __shfl_sync(0xffffffffu, (uint32_t)(uint16_t)P.fallback | ((uint32_t)(uint16_t)P.narrow << 16), 0);
    P.fallback = (int16_t)(f & 0xFFFFu);
    P.narrow = (int16_t)(f >> 16);
  } else {
    const uint32_t wid = rank >> 5;
    if (lane == 0) {
      sm->S[wid] = S;
      sm->mx[wid] = mx;
      sm->mn[wid] = mn;
    }
    group_sync(bar_id, GROUP);
    if (rank == 0) {
      for (int k = 1; k < GROUP / 32; k++) {
        S += sm->S[k];
        mx = max(mx, sm->mx[k]);
        mn = min(mn, sm->mn[k]);
      }
      sm->P = solve(S);
    }
    group_sync(bar_id, GROUP);
    P = sm->P;
  }

  // pass 2
  int64_t lo = INT64_MAX, hi = INT64_MIN;
  uint64_t zmax = 0;
  if (P.fallback) {
    for (uint32_t x = rank; x < N; x += GROUP) {
      const uint64_t v = u32 ? (uint64_t)__ldg(v32 + x) : __ldg(v64 + x);
      zmax = max(zmax, zz_encode((int64_t)(v - (uint64_t)P.fb_shift)));
    }
    if (GROUP > 1) zmax = warp_max_u64(zmax);
  } else {
    if (u32)
      fit_pass2<GROUP>(v32, N, P, rank, &lo, &hi);
    else
      fit_pass2<GROUP>(v64, N, P, rank, &lo, &hi);
    if (GROUP > 1) {
      lo = warp_min_i64(lo);
      hi = warp_max_i64(hi);
    }
  }
  FitResult R;
  if (GROUP == 1) {
    R = finish_fit(P, lo, hi, zmax);
  } else if (GROUP == 32) {
    if (lane == 0) R = finish_fit(P, lo, hi, zmax);
    R.theta0 = __shfl_sync(0xffffffffu, R.theta0, 0);
    R.theta1 = __shfl_sync(0xffffffffu, R.theta1, 0);
    R.s = __shfl_sync(0xffffffffu, R.s, 0);
    R.b = __shfl_sync(0xffffffffu, R.b, 0);
  } else {
    const uint32_t wid = rank >> 5;
    if (lane == 0) {
      sm->mx[wid] = hi;
      sm->mn[wid] = lo;
      sm->zmax[wid] = zmax;
    }
    group_sync(bar_id, GROUP);
    if (rank == 0) {
      for (int k = 1; k < GROUP / 32; k++) {
        hi = max(hi, sm->mx[k]);
        lo = min(lo, sm->mn[k]);
        zmax = max(zmax, sm->zmax[k]);
      }
      sm->R = finish_fit(P, lo, hi, zmax);
    }
    group_sync(bar_id, GROUP);
    R = sm->R;
    group_sync(bar_id, GROUP);  // sm is reused by the next partition
  }
  return R;
}

// minimum, maximum and sum over aligned tiles of TILE lanes (32: the warp), in every lane
template <int TILE>
__device__ __forceinline__ int32_t tile_min(int32_t v) {
  if constexpr (TILE == 32) {
    v = __reduce_min_sync(0xffffffffu, v);
  } else {
    for (int o = TILE / 2; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}
template <int TILE>
__device__ __forceinline__ int32_t tile_max(int32_t v) {
  if constexpr (TILE == 32) {
    v = __reduce_max_sync(0xffffffffu, v);
  } else {
    for (int o = TILE / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  }
  return v;
}
template <int TILE>
__device__ __forceinline__ int64_t tile_min(int64_t v) {
  for (int o = TILE / 2; o > 0; o >>= 1) v = min(v, (int64_t)__shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int TILE>
__device__ __forceinline__ int64_t tile_max(int64_t v) {
  for (int o = TILE / 2; o > 0; o >>= 1) v = max(v, (int64_t)__shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int TILE>
__device__ __forceinline__ uint64_t tile_max(uint64_t v) {
  for (int o = TILE / 2; o > 0; o >>= 1) v = max(v, (uint64_t)__shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int TILE>
__device__ __forceinline__ int64_t tile_sum(int64_t v) {
  for (int o = TILE / 2; o > 0; o >>= 1) v += (int64_t)__shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Fit of one short partition per tile of TILE lanes (N = 0: the tile only takes part in the warp's steps), r
// the lane's place in it; the result in every lane. A warp that fits one partition at a time spends as long in
// its one-lane solve as on 256 values; here 32 / TILE partitions solve at once and their loads are in flight
// together.
template <int TILE, typename T>
__device__ __forceinline__ FitResult fit_tile(const T* __restrict__ v, uint32_t N, int model, uint32_t r) {
  const bool lin = model == LECO_MODEL_LINEAR && N >= 2;
  const int64_t ref = N ? (int64_t)__ldg(v) : 0;
  int32_t mx32 = 0, mn32 = 0, u = 2 * (int32_t)r - ((int32_t)N - 1);
  uint32_t far = 0;
  int64_t sum = 0;
  auto always = []() { return true; };
  for_runs<TILE, 8>(
      v, N, r, (T)ref,
      [&](T value) {
        const int64_t d = (int64_t)value - ref;
        const int32_t e = (int32_t)d;
        far |= (uint32_t)((int32_t)(d >> 32) ^ (e >> 31));  // d outside 32 bits
        mx32 = max(mx32, e);
        mn32 = min(mn32, e);
        sum += (int64_t)u * e;
        u += 2 * TILE;
      },
      always);
  i128 S;
  int64_t mx, mn;
  if (__all_sync(0xffffffffu, far == 0 && mn32 > -(int32_t)kNarrow && mx32 < (int32_t)kNarrow && narrow_ref(ref))) {
    S = tile_sum<TILE>(sum);
    mx = ref + tile_max<TILE>(mx32);
    mn = ref + tile_min<TILE>(mn32);
  } else {
    fit_pass1_wide<TILE>(v, N, lin, r, &S, &mx, &mn);
    for (int o = TILE / 2; o > 0; o >>= 1) {
      const uint64_t lo = __shfl_xor_sync(0xffffffffu, (uint64_t)S, o), hi = __shfl_xor_sync(0xffffffffu, (uint64_t)((u128)S >> 64), o);
      S += (i128)(((u128)hi << 64) | lo);
    }
    mx = tile_max<TILE>(mx);
    mn = tile_min<TILE>(mn);
  }
  FitParams P;
  P.B = 0;
  P.fb_shift = 0;
  P.s = 0;
  P.fallback = 0;
  P.narrow = 1;
  if (N) {
    P = solve_params(lin ? S : (i128)0, mx, mn, N, lin);
    P.narrow = narrow_line(P, N) && narrow_ref(mn) && narrow_diff(mx - mn) ? 1 : 0;
  }
  int64_t lo = INT64_MAX, hi = INT64_MIN;
  uint64_t zmax = 0;
  if (__all_sync(0xffffffffu, P.narrow)) {
    int32_t l, h;
    fit_pass2_narrow<TILE>(v, N, P.B, P.s, r, ref, &l, &h);
    lo = ref + tile_min<TILE>(l);
    hi = ref + tile_max<TILE>(h);
  } else {
    if (P.fallback) {
      for (uint32_t x = r; x < N; x += TILE) zmax = max(zmax, zz_encode((int64_t)((uint64_t)__ldg(v + x) - (uint64_t)P.fb_shift)));
    } else {
      P.narrow = 0;
      fit_pass2<TILE>(v, N, P, r, &lo, &hi);
    }
    lo = tile_min<TILE>(lo);
    hi = tile_max<TILE>(hi);
    zmax = tile_max<TILE>(zmax);
  }
  return finish_fit(P, lo, hi, zmax);
}

// ------------------------------------------------------------------------------ polynomial model
//
// §3.1 names polynomial terms among the model family; §4 chooses per partition among constant,
// linear and polynomials up to degree three. This fit follows one exact reading of that choice:
//  1. one pass: min, max, and S_j = sum p_j(x) w_x (j = 1..3) over the Gram polynomials of the
//     partition, p1 = x', p2 = 3x'^2 - (N^2-1), p3 = 5x'^3 - (3N^2-7)x' with x' = 2x - (N-1); the p_j
//     are orthogonal to 1 and to each other over x < N, so S_j / |p_j|^2 is the least-squares
//     coefficient c_j of p_j for any degree that includes it (and S_1 is the line's moment);
//  2. a thread solves the constant and linear parameters (as for those models) and, when
//     64 <= N <= 16384 and max - min < 2^62, the quadratic and cubic grids: c_j as one binary64
//     division of the two integers (each converted from sign and magnitude), s_j = min(62, 61 - e_j)
//     with |c_j| < 2^e_j, S = max s_j capped so that every K_j 2^(S - s_j) p_j stays below 2^124,
//     K_j = round(c_j 2^s_j) half up;
//  3. a second pass: the linear residual range (or the fallback's widest zigzag residual) and, per
//     polynomial, the range of w_x - floor(F(x) / 2^S) (F = sum K_j 2^(S - s_j) p_j(x), exact);
//  4. a thread sizes the four candidates (256 + N b for constant and linear, 576 + N b for the
//     polynomials, whose minimax intercept T and width follow from their range as for the line) and
//     keeps the smallest, ties to the earlier.

// headroom (bits) of K_j 2^(S - s_j) p_j below 2^124: |K_j| <= 2^61, |p_j| < 2^14, 2^29, 2^43
__host__ __device__ constexpr int32_t poly_headroom(int j) { return j == 1 ? 49 : (j == 2 ? 34 : 20); }

// |p_j|^2 over N points: N(N^2-1)/3, 4N(N^2-1)(N^2-4)/5, 4N(N^2-1)(N^2-4)(N^2-9)/7
__device__ __forceinline__ i128 gram_norm(int j, uint32_t N) {
  const i128 n = N, n2 = n * n;
  const i128 base = n * (n2 - 1);
  if (j == 1) return floordiv_i128(base, 3);
  if (j == 2) return floordiv_i128(4 * base * (n2 - 4), 5);
  return floordiv_i128(4 * base * (n2 - 4) * (n2 - 9), 7);
}

// binary64 from sign and magnitude: +-(double(hi) 2^64 + double(lo)), each step rounded to nearest
__device__ __forceinline__ double i128_to_f64(i128 v) {
  const u128 mag = v < 0 ? (u128)0 - (u128)v : (u128)v;
  const double d = __dadd_rn(__dmul_rn(__ull2double_rn((uint64_t)(mag >> 64)), 18446744073709551616.0),
                             __ull2double_rn((uint64_t)mag));
  return v < 0 ? -d : d;
}

// F(x) = sum_j K_j 2^(S - s_j) p_j(x) expanded in powers of the local index x (all exact):
// p1 = 2x + (1-N), p2 = 12x^2 + (12-12N)x + (2N^2-6N+4),
// p3 = 40x^3 + (60-60N)x^2 + (24N^2-60N+44)x + (-2N^3+12N^2-22N+12).
__host__ __device__ __forceinline__ PolyAux poly_aux_from(const int64_t* K, const int32_t* sj, int32_t S, uint32_t N) {
  const i128 n = N;
  const i128 G1 = (i128)K[0] * ((i128)1 << (S - sj[0]));
  const i128 G2 = (i128)K[1] * ((i128)1 << (S - sj[1]));
  const i128 G3 = (i128)K[2] * ((i128)1 << (S - sj[2]));
  i128 a[4];
  a[3] = 40 * G3;
  a[2] = 12 * G2 + (60 - 60 * n) * G3;
  a[1] = 2 * G1 + (12 - 12 * n) * G2 + (24 * n * n - 60 * n + 44) * G3;
  a[0] = (1 - n) * G1 + (2 * n * n - 6 * n + 4) * G2 + (-2 * n * n * n + 12 * n * n - 22 * n + 12) * G3;
  PolyAux r;
  for (int k = 0; k < 4; k++) {
    r.a[k][0] = (uint64_t)(u128)a[k];
    r.a[k][1] = (uint64_t)((u128)a[k] >> 64);
  }
  return r;
}

// The cubic F(x) = c0 + c1 x + c2 x^2 + c3 x^3 (128-bit, from a PolyAux row) at x and its forward
// differences over the stride h, each multiplied by 2^up modulo 2^128:
// D1 = c1 h + c2 (2xh + h^2) + c3 (3x^2 h + 3x h^2 + h^3), D2 = c2 2h^2 + c3 (6x h^2 + 6h^3),
// D3 = c3 6h^3 (x and h below 2^14 and 2^8 keep every bracket inside 64 bits). Stepping
// F += D1, D1 += D2, D2 += D3 then gives F at x + h, x + 2h, ... exactly (modulo 2^128).
struct PolySteps {
  u128 F, D1, D2, D3;
};

__device__ __forceinline__ PolySteps poly_steps(const PolyAux& q, uint64_t x, uint64_t h, uint32_t up) {
  u128 c[4];
  for (int k = 0; k < 4; k++) c[k] = ((u128)q.a[k][1] << 64) | q.a[k][0];
  PolySteps r;
  r.F = (((c[3] * x + c[2]) * x + c[1]) * x + c[0]) << up;
  r.D1 = (c[1] * h + c[2] * (2 * x * h + h * h) + c[3] * (3 * x * x * h + 3 * x * h * h + h * h * h)) << up;
  r.D2 = (c[2] * (2 * h * h) + c[3] * (6 * x * h * h + 6 * h * h * h)) << up;
  r.D3 = (c[3] * (6 * h * h * h)) << up;
  return r;
}

__device__ __forceinline__ void poly_step(PolySteps& r) {
  r.F += r.D1;
  r.D1 += r.D2;
  r.D2 += r.D3;
}

// one polynomial candidate's grid (step 2)
struct PolyGrid {
  int64_t K[3];
  int32_t sj[3];
  int32_t S;
  int32_t valid;
};

__device__ PolyGrid poly_grid(const i128* Sm, uint32_t N, int degree) {
  PolyGrid g;
  g.valid = 0;
  g.S = 0;
  double c[3] = {0.0, 0.0, 0.0};
  int32_t cap = 1 << 30;
  for (int j = 0; j < 3; j++) {
    g.K[j] = 0;
    g.sj[j] = 0;
  }
  for (int j = 0; j < degree; j++) {
    c[j] = __ddiv_rn(i128_to_f64(Sm[j]), i128_to_f64(gram_norm(j + 1, N)));
    if (c[j] != 0.0) {
      int e;
      frexp(c[j], &e);  // |c| < 2^e
      int32_t sj = 61 - e;
      if (sj > 62) sj = 62;
      if (sj < 0) return g;
      g.sj[j] = sj;
      g.S = max(g.S, sj);
      cap = min(cap, sj + poly_headroom(j + 1));
    }
  }
  g.S = min(g.S, cap);
  for (int j = 0; j < degree; j++) {
    g.sj[j] = min(g.sj[j], g.S);
    const double y = __dmul_rn(c[j], pow2(g.sj[j]));  // exact: a power-of-two scale
    const double f = floor(y);
    g.K[j] = __double2ll_rz(f) + (__dsub_rn(y, f) >= 0.5 ? 1 : 0);
  }
  g.valid = 1;
  return g;
}

// What the polynomial model chose for one partition: kind 0 constant, 1 linear (R: the record's
// theta, s and b exactly as those models write them), 2 quadratic, 3 cubic (pc: its block).
struct FitChoice {
  FitResult R;
  PolyCoef pc;
  uint32_t kind;
  uint32_t b;
};

// The polynomial model's fit runs as four phases, each its own kernel so that none carries the
// others' registers: moments (a warp per partition), plan (a thread: every candidate's parameters),
// ranges (a warp: the residual ranges under them), choice (a thread: sizes and the record).

// phase 1 result: min, max and the Gram moments S_j = sum p_j(x) w_x (S_1 is the line's moment)
struct PolyMom {
  i128 S[3];
  int64_t mx, mn;
};
static_assert(sizeof(PolyMom) == 64, "poly moments layout");

// phase 2 result
struct PolyPlan {
  FitParams PC, PL;  // constant and linear parameters (as those models solve them)
  PolyGrid G[2];     // quadratic and cubic grids (valid = 0: the candidate does not apply)
  PolyAux Q[2];      // their F as 128-bit monomial coefficients
  int32_t fast[2];   // |floor(F / 2^S)| is bounded so that every residual fits int64 (see poly_plan)
  int32_t narrow;    // values within 2^30 of each other; the line and every valid polynomial within 2^30
  int32_t pad;
};

// phase 3 result
struct PolyRange {
  int64_t lo, hi;   // the line's residual range (not fallback)
  uint64_t zmax;    // the fallback's widest zigzag residual
  int64_t plo[2], phi[2];
  int32_t bad[2];   // a residual outside int64: the candidate does not apply
};

__device__ __forceinline__ int64_t poly_value_at(const uint32_t* v32, const uint64_t* v64, bool u32, uint32_t x) {
  return u32 ? (int64_t)__ldg(v32 + x) : (int64_t)__ldg(v64 + x);
}

// phase 1 of a narrow partition of at least kPolyMinLen values by one warp (the result in every lane). The
// Gram polynomials sum to zero over the partition, so S_j = sum p_j(x) d_x with d_x = w_x - w_0 in 32 bits. A
// lane's positions x = c + lane + 32 k, k < 128, give power sums M_i = sum k^i d (k^3 < 2^21,
// d < 2^30, 128 terms: below 2^58), three 32 x 32 -> 64-bit products per value; with x' = X + 64 k, the lane then
// expands p_1 = x', p_2 = 3 x'^2 - (N^2 - 1) and p_3 = 5 x'^3 - (3 N^2 - 7) x' in k once per 128 values, in 128 bits.
// 50M values in partitions of 4096: 262 -> 109 us against three 128-bit products per value.
template <typename T>
__device__ __forceinline__ bool poly_moments_narrow(const T* __restrict__ v, uint32_t N, uint32_t lane, int64_t ref,
                                                    PolyMom& M) {
  if (!narrow_ref(ref)) return false;
  int32_t mx = 0, mn = 0;
  uint32_t far = 0;
  i128 S[3] = {0, 0, 0};
  const int64_t A2 = (int64_t)N * N - 1, A3 = 3 * (int64_t)N * N - 7;
  for (uint32_t c = 0; c < N; c += 4096) {
    const uint32_t n = min(N - c, 4096u);
    int64_t M0 = 0, M1 = 0, M2 = 0, M3 = 0;
    int32_t k = 0;
    for_runs<32, 8>(
        v + c, n, lane, (T)ref,
        [&](T value) {
          const int64_t d = (int64_t)value - ref;
          const int32_t e = (int32_t)d;
          far |= (uint32_t)((int32_t)(d >> 32) ^ (e >> 31));  // d outside 32 bits
          mx = max(mx, e);
          mn = min(mn, e);
          M0 += e;
          M1 += (int64_t)k * e;
          M2 += (int64_t)(k * k) * e;
          M3 += (int64_t)(k * k * k) * e;
          k++;
        },
        []() { return true; });
    if (__any_sync(0xffffffffu, far != 0 || mn <= -(int32_t)kNarrow || mx >= (int32_t)kNarrow)) return false;
    const int64_t X = 2 * ((int64_t)lane + c) - ((int64_t)N - 1);
    S[0] += mul_s64(X, M0) + 64 * (i128)M1;
    S[1] += mul_s64(3 * X * X - A2, M0) + mul_s64(384 * X, M1) + mul_s64(12288, M2);
    S[2] += mul_s64((5 * X * X - A3) * X, M0) + mul_s64(960 * X * X - 64 * A3, M1) + mul_s64(61440 * X, M2) +
            mul_s64(1310720, M3);
  }
  for (int j = 0; j < 3; j++) M.S[j] = warp_sum_i128(S[j]);
  M.mx = ref + __reduce_max_sync(0xffffffffu, mx);
  M.mn = ref + __reduce_min_sync(0xffffffffu, mn);
  return true;
}

// phase 1 by one warp; the result in lane 0
__device__ PolyMom poly_moments_warp(const void* __restrict__ values, int dtype, uint64_t a, uint32_t N,
                                     uint32_t lane) {
  const bool u32 = dtype == LECO_U32;
  const uint32_t* v32 = static_cast<const uint32_t*>(values) + a;
  const uint64_t* v64 = static_cast<const uint64_t*>(values) + a;
  const bool poly_len = N >= kPolyMinLen && N <= kPolyMaxLen;
  PolyMom M;
  if (poly_len && (u32 ? poly_moments_narrow(v32, N, lane, (int64_t)__ldg(v32), M)
                       : poly_moments_narrow(v64, N, lane, (int64_t)__ldg(v64), M)))
    return M;
  int64_t mx = INT64_MIN, mn = INT64_MAX;
  i128 Sm[3] = {0, 0, 0};
  const int64_t nm1 = (int64_t)N - 1;
  const int64_t n2m1 = (int64_t)N * N - 1, c3 = 3 * (int64_t)N * N - 7;
  for (uint32_t x = lane; x < N; x += 32) {
    const int64_t w = poly_value_at(v32, v64, u32, x);
    mx = max(mx, w);
    mn = min(mn, w);
    const int64_t xp = 2 * (int64_t)x - nm1;
    Sm[0] += (i128)xp * w;
    if (poly_len) {
      const int64_t xp2 = xp * xp;
      Sm[1] += (i128)(3 * xp2 - n2m1) * w;
      Sm[2] += (i128)((5 * xp2 - c3) * xp) * w;
    }
  }
  for (int j = 0; j < 3; j++) M.S[j] = warp_sum_i128(Sm[j]);
  M.mx = warp_max_i64(mx);
  M.mn = warp_min_i64(mn);
  return M;
}

// phase 2 (one thread)
__device__ PolyPlan poly_plan(const PolyMom& M, uint32_t N) {
  PolyPlan P;
  P.PC = solve_params(M.S[0], M.mx, M.mn, N, false);
  P.PL = solve_params(M.S[0], M.mx, M.mn, N, N >= 2);
  const bool elig = N >= kPolyMinLen && N <= kPolyMaxLen && (i128)M.mx - (i128)M.mn < ((i128)1 << 62);
  P.narrow = elig && narrow_line(P.PL, N) && narrow_ref(M.mn) && narrow_diff(M.mx - M.mn) ? 1 : 0;
  for (int d = 0; d < 2; d++) {
    P.G[d].valid = 0;
    P.fast[d] = 0;
    if (elig) P.G[d] = poly_grid(M.S, N, 2 + d);
    if (!P.G[d].valid) continue;
    P.Q[d] = poly_aux_from(P.G[d].K, P.G[d].sj, P.G[d].S, N);
    // |F(x)| <= sum_j |K_j| 2^(S - s_j) max|p_j| with max|p_1| < N, max|p_2| <= 2N^2, max|p_3| <= 2N^3;
    // with q = floor(F / 2^S) in [-Bq, Bq], every residual w - q lies in [mn - Bq, mx + Bq]
    const u128 n = N;
    const u128 bnd[3] = {n, 2 * n * n, 2 * n * n * n};
    u128 Fb = 0;
    for (int j = 0; j < 3; j++) {
      const int64_t k = P.G[d].K[j];
      const u128 ak = (u128)(k < 0 ? -(i128)k : (i128)k) << (P.G[d].S - P.G[d].sj[j]);
      Fb += ak * bnd[j];
    }
    const i128 Bq = (i128)(Fb >> P.G[d].S) + 1;
    P.fast[d] = Bq < ((i128)1 << 62) && (i128)M.mn - Bq > (i128)INT64_MIN && (i128)M.mx + Bq < (i128)INT64_MAX;
    if (Bq >= (i128)kNarrow) P.narrow = 0;
  }
  return P;
}

// phase 3 of a narrow plan by one warp (the result in every lane). The residual w - floor(y) is ceil(w - y) and
// ceil is monotone, so the extremes of the residuals are the ceilings of the extremes of w - y: y = F / 2^S is
// stepped in 32.32 fixed point (F's forward differences over 32 positions, each truncated to 2^-32) and only the
// extremes of (w - w_0) - y are kept, 16 instructions per polynomial and value where the exact 128-bit steps take
// 40. After k steps the truncations add up to less than (C(k,3) + C(k,2) + k + 1) 2^-32; an extreme
// closer than that to an integer leaves the partition to the exact pass. With four extremes (k <= 512) that is up to
// one partition in 48 at 16384 values and one in 3000 at 4096, and every one whose residuals are whole numbers
// (values on an integer polynomial without noise), which takes both passes. 50M values in partitions of 4096:
// 319 -> 183 us.
template <typename T>
__device__ __forceinline__ bool poly_ranges_narrow(const T* __restrict__ v, uint32_t N, uint32_t lane, int64_t ref,
                                                   const PolyPlan* __restrict__ plan, PolyRange& R) {
  const NarrowLine line(plan->PL.B, plan->PL.s);
  int32_t l = INT32_MAX, h = INT32_MIN;
  uint64_t G = line.B * lane;
  const uint64_t dG = line.B * 32u;
  uint64_t F[2], D1[2], D2[2], D3[2];  // modulo 2^64: |y| < 2^30
  int64_t lo[2] = {INT64_MAX, INT64_MAX}, hi[2] = {INT64_MIN, INT64_MIN};
  bool valid[2];
#pragma unroll
  for (int d = 0; d < 2; d++) {
    valid[d] = plan->G[d].valid != 0;
    F[d] = D1[d] = D2[d] = D3[d] = 0;
    if (!valid[d]) continue;
    const int32_t S = plan->G[d].S;
    const PolySteps q = poly_steps(plan->Q[d], lane, 32, 0);
    auto fix = [&](u128 x) { return (uint64_t)(S >= 32 ? (i128)x >> (S - 32) : (i128)(x << (32 - S))); };
    F[d] = fix(q.F);
    D1[d] = fix(q.D1);
    D2[d] = fix(q.D2);
    D3[d] = fix(q.D3);
  }
  const uint32_t r32 = (uint32_t)ref;
  for_runs<32, 4>(
      v, N, lane, (T)ref,
      [&](T value) {
        const int32_t e = (int32_t)((uint32_t)value - r32);
        const int32_t r = e - line.at(G);
        l = min(l, r);
        h = max(h, r);
        G += dG;
#pragma unroll
        for (int d = 0; d < 2; d++) {
          const int64_t y = (int64_t)(((uint64_t)(uint32_t)e << 32) - F[d]);
          lo[d] = min(lo[d], y);
          hi[d] = max(hi[d], y);
          F[d] += D1[d];
          D1[d] += D2[d];
          if (d == 1) D2[d] += D3[d];
        }
      },
      []() { return true; });
  R.lo = ref + __reduce_min_sync(0xffffffffu, l);
  R.hi = ref + __reduce_max_sync(0xffffffffu, h);
  R.zmax = 0;
  const uint64_t k = (N + 31) / 32;
  const int64_t err = (int64_t)(k * k * k / 6 + k * k / 2 + k + 2);
  bool sure = true;
  for (int d = 0; d < 2; d++) {
    R.plo[d] = INT64_MAX;
    R.phi[d] = INT64_MIN;
    R.bad[d] = 0;
    if (!valid[d]) continue;
    // every truncation lowers F, so the true y of a position is in (y - err, y]
    const int64_t a = tile_min<32>(lo[d]), b = tile_max<32>(hi[d]);
    auto up = [](int64_t y) { return (y + (int64_t)0xFFFFFFFF) >> 32; };  // ceil(y / 2^32)
    sure = sure && up(a - err) == up(a) && up(b - err) == up(b);
    R.plo[d] = ref + up(a);
    R.phi[d] = ref + up(b);
  }
  return sure;
}

// phase 3 by one warp; the result in lane 0. One pass: the line's residual (or the fallback's
// zigzag residual) and both polynomials' residuals at the lane's positions x = lane + 32k, each
// polynomial's F by forward differences over the stride 32 (exact 128-bit; x < 2^14, so every
// bracket fits 64 bits).
__device__ PolyRange poly_ranges_warp(const void* __restrict__ values, int dtype, uint64_t a, uint32_t N,
                                      uint32_t lane, const PolyPlan* __restrict__ plan) {
  const bool u32 = dtype == LECO_U32;
  const uint32_t* v32 = static_cast<const uint32_t*>(values) + a;
  const uint64_t* v64 = static_cast<const uint64_t*>(values) + a;
  PolyRange R;
  if (plan->narrow && (u32 ? poly_ranges_narrow(v32, N, lane, (int64_t)__ldg(v32), plan, R)
                           : poly_ranges_narrow(v64, N, lane, (int64_t)__ldg(v64), plan, R)))
    return R;
  const int64_t B = plan->PL.B, fb = plan->PL.fb_shift;
  const int32_t s = plan->PL.s, fallback = plan->PL.fallback;
  bool valid[2], fast[2];
  int32_t S[2];
  PolySteps Fd[2];
  for (int d = 0; d < 2; d++) {
    valid[d] = plan->G[d].valid != 0;
    fast[d] = valid[d] && plan->fast[d];
    S[d] = plan->G[d].S;
    // fast: carried times 2^(64-S) modulo 2^128, so that floor(F / 2^S) mod 2^64 (= floor(F / 2^S),
    // which the plan bounded inside int64) is the high half
    const uint32_t up = fast[d] ? 64u - (uint32_t)S[d] : 0u;
    Fd[d] = valid[d] ? poly_steps(plan->Q[d], lane, 32, up) : PolySteps{0, 0, 0, 0};
  }
  int64_t lo = INT64_MAX, hi = INT64_MIN;
  uint64_t zmax = 0;
  int64_t plo[2] = {INT64_MAX, INT64_MAX}, phi[2] = {INT64_MIN, INT64_MIN};
  int bad[2] = {0, 0};
  for (uint32_t x = lane; x < N; x += 32) {
    const int64_t w = poly_value_at(v32, v64, u32, x);
    if (fallback) {
      zmax = max(zmax, zz_encode((int64_t)((uint64_t)w - (uint64_t)fb)));
    } else {
      const uint64_t Fl = (uint64_t)B * x;
      const int64_t r = w - (s >= 0 ? ((int64_t)Fl >> s) : (int64_t)(Fl << (-s)));
      lo = min(lo, r);
      hi = max(hi, r);
    }
#pragma unroll
    for (int d = 0; d < 2; d++) {
      if (!valid[d]) continue;
      if (fast[d]) {
        const int64_t r = w - (int64_t)(uint64_t)(Fd[d].F >> 64);
        plo[d] = min(plo[d], r);
        phi[d] = max(phi[d], r);
      } else {
        const i128 r = (i128)w - ((i128)Fd[d].F >> S[d]);
        if (r > (i128)INT64_MAX || r < (i128)INT64_MIN) {
          bad[d] = 1;
        } else {
          plo[d] = min(plo[d], (int64_t)r);
          phi[d] = max(phi[d], (int64_t)r);
        }
      }
      poly_step(Fd[d]);
    }
  }
  R.lo = warp_min_i64(lo);
  R.hi = warp_max_i64(hi);
  R.zmax = warp_max_u64(zmax);
  for (int d = 0; d < 2; d++) {
    R.plo[d] = warp_min_i64(plo[d]);
    R.phi[d] = warp_max_i64(phi[d]);
    R.bad[d] = __any_sync(0xffffffffu, bad[d]);
  }
  return R;
}

// phase 4 (one thread): size the four candidates (256 + N b for constant and linear, 576 + N b for
// the polynomials, whose minimax intercept and width follow from their range as for the line) and
// keep the smallest, ties to the earlier
__device__ FitChoice poly_choose(const PolyMom& M, const PolyPlan& P, const PolyRange& R, uint32_t N) {
  FitChoice C;
  C.R = finish_fit(P.PC, M.mn, M.mx, R.zmax);  // a constant fallback implies the linear one: same zmax
  C.kind = 0;
  C.b = C.R.b;
  uint64_t best = kSmBits + (uint64_t)N * C.R.b;
  const FitResult RL = finish_fit(P.PL, R.lo, R.hi, R.zmax);
  if (kSmBits + (uint64_t)N * RL.b < best) {
    best = kSmBits + (uint64_t)N * RL.b;
    C.R = RL;
    C.kind = 1;
    C.b = RL.b;
  }
  for (int d = 0; d < 2; d++) {
    if (!P.G[d].valid || R.bad[d]) continue;
    const i128 t = (i128)R.plo[d] + (((i128)R.phi[d] - (i128)R.plo[d] + 1) >> 1);
    const uint64_t z = max(zz_encode((int64_t)((i128)R.plo[d] - t)), zz_encode((int64_t)((i128)R.phi[d] - t)));
    const uint32_t b = (uint32_t)bitlen_u64(z);
    const uint64_t size = kSmBits + kPolyBlockBits + (uint64_t)N * b;
    if (size < best) {
      best = size;
      C.kind = 2 + d;
      C.b = b;
      C.pc.T = (int64_t)t;
      for (int j = 0; j < 3; j++) C.pc.K[j] = P.G[d].K[j];
      C.pc.E = (uint64_t)P.G[d].sj[0] | ((uint64_t)P.G[d].sj[1] << 8) | ((uint64_t)P.G[d].sj[2] << 16);
    }
  }
  return C;
}

}  // namespace
}  // namespace leco
