// Encoder kernels (§3.1 Regressor, §3.3 Encoder): per-partition fit (fit.cuh), offset scan,
// decode-table build and residual packing.
#include <type_traits>

#include "fit.cuh"
#include "launch_shape.cuh"
#include "leco_internal.cuh"

namespace leco {

namespace {

constexpr int kFitBlock = 256;
constexpr int kFitWarps = kFitBlock / 32;
// CTAs of kFitBlock threads per SM for the fit (registers capped to fit them): the fit is bound by
// instruction issue, so more resident warps beat keeping every partition in flight inside L2
constexpr int kFitCtasPerSm = 4;

__device__ __forceinline__ uint64_t part_begin(const uint64_t* starts, uint32_t L, uint64_t n,
                                               uint64_t p) {
  if (starts) return starts[p];
  const uint64_t s = p * (uint64_t)L;
  return s < n ? s : n;
}

// the record of a fitted partition [a, a + N), its stream bits and the column's widest width
__device__ __forceinline__ void put_fit(const FitResult& R, uint64_t a, uint32_t N, uint64_t p, Record* __restrict__ rec,
                                        uint64_t* __restrict__ lenbits, uint32_t* __restrict__ max_b) {
  Record r;
  r.theta0 = R.theta0;
  r.theta1 = R.theta1;
  r.start = a;
  r.word3 = make_w3(0, R.b, R.s, 1);
  rec[p] = r;
  lenbits[p] = (uint64_t)N * R.b;
  if (R.b) atomicMax(max_b, R.b);
}

// Tiles of TILE lanes per partition (fixed partitions below 1024 values), or a warp (TILE = 32: partitions of
// any lengths), grid-stride: reductions are shuffles, the second pass re-reads the partition from L1 or L2.
template <typename T, int TILE>
__global__ void __launch_bounds__(kFitBlock, kFitCtasPerSm)
    k_fit(const T* __restrict__ values, uint64_t n, const uint64_t* __restrict__ starts, uint32_t L, uint64_t m,
          int model, Record* __restrict__ rec, uint64_t* __restrict__ lenbits, uint32_t* __restrict__ max_b) {
  constexpr uint32_t kTiles = 32 / TILE;
  const uint32_t lane = threadIdx.x & 31u, r = lane % TILE;
  const uint64_t nw = (uint64_t)gridDim.x * kFitWarps;
  for (uint64_t p0 = ((uint64_t)blockIdx.x * kFitWarps + (threadIdx.x >> 5)) * kTiles; p0 < m; p0 += nw * kTiles) {
    const uint64_t p = p0 + lane / TILE;
    uint64_t a = 0;
    uint32_t N = 0;
    if (p < m) {
      a = part_begin(starts, L, n, p);
      N = (uint32_t)(part_begin(starts, L, n, p + 1) - a);
    }
    FitResult R;
    if (TILE == 32)
      R = fit_range<32>(values, sizeof(T) == 4 ? LECO_U32 : LECO_U64, a, N, model, lane, nullptr);
    else
      R = fit_tile<TILE>(values + a, N, model, r);
    if (r == 0 && N) put_fit(R, a, N, p, rec, lenbits, max_b);
  }
}

// Many short partitions of any lengths: a warp takes four, a tile of eight lanes each when all have at most
// kFitShortVals values, else one after another. A warp per partition spends as long in its one-lane solve as on 256
// values: 2.7M partitions of 1 .. 15 values 2.15 -> 0.54 ms, 400K of 1 .. 99 355 -> 102 us. Not for columns whose
// mean is above kFitShortMean: beside this path the warp's own is slower (partitions of 1 .. 999 values 57 -> 70 us).
constexpr uint32_t kFitShortVals = 256, kFitShortMean = 128;

template <typename T>
__global__ void __launch_bounds__(kFitBlock, kFitCtasPerSm)
    k_fit_short(const T* __restrict__ values, uint64_t n, const uint64_t* __restrict__ starts, uint64_t m, int model,
                Record* __restrict__ rec, uint64_t* __restrict__ lenbits, uint32_t* __restrict__ max_b) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nw = (uint64_t)gridDim.x * kFitWarps;
  for (uint64_t p0 = ((uint64_t)blockIdx.x * kFitWarps + (threadIdx.x >> 5)) * 4; p0 < m; p0 += nw * 4) {
    const uint64_t p = p0 + lane / 8;
    uint64_t a = 0;
    uint32_t N = 0;
    if (p < m) {
      a = starts[p];
      N = (uint32_t)(starts[p + 1] - a);
    }
    if (__all_sync(0xffffffffu, N <= kFitShortVals)) {
      const FitResult R = fit_tile<8>(values + a, N, model, lane & 7u);
      if ((lane & 7u) == 0 && N) put_fit(R, a, N, p, rec, lenbits, max_b);
      continue;
    }
    for (int k = 0; k < 4; k++) {
      const uint64_t ak = __shfl_sync(0xffffffffu, a, 8 * k);
      const uint32_t nk = __shfl_sync(0xffffffffu, N, 8 * k);
      if (nk == 0) break;  // past the last partition
      const FitResult R = fit_range<32>(values, sizeof(T) == 4 ? LECO_U32 : LECO_U64, ak, nk, model, lane, nullptr);
      if (lane == 0) put_fit(R, ak, nk, p0 + k, rec, lenbits, max_b);
    }
  }
}

// Two warps per partition (four partitions per 256-thread CTA, each pair of warps synchronised by its
// own named barrier): as many warps stream as with one warp per partition, but half as many
// partitions are in flight, so the second pass finds the partition in L2 instead of DRAM.
constexpr int kFitPairs = kFitBlock / 64;
constexpr int kPairCtas = 3;  // sixteen loads in flight per lane need the registers (4 CTAs: 1081 us a pass, 3: 1061)

__global__ void __launch_bounds__(kFitBlock, kPairCtas)
    k_fit_pairs(const void* __restrict__ values, int dtype, uint64_t n, const uint64_t* __restrict__ starts,
                uint32_t L, uint64_t m, int model, Record* __restrict__ rec, uint64_t* __restrict__ lenbits,
                uint32_t* __restrict__ max_b) {
  __shared__ FitShared sm[kFitPairs];
  const uint32_t g = threadIdx.x >> 6, rank = threadIdx.x & 63u;
  const uint64_t ng = (uint64_t)gridDim.x * kFitPairs;
  for (uint64_t p = (uint64_t)blockIdx.x * kFitPairs + g; p < m; p += ng) {
    const uint64_t a = part_begin(starts, L, n, p);
    const uint32_t N = (uint32_t)(part_begin(starts, L, n, p + 1) - a);
    const FitResult R = fit_range<64>(values, dtype, a, N, model, rank, &sm[g], 1 + (int)g);
    if (rank == 0) put_fit(R, a, N, p, rec, lenbits, max_b);
  }
}

// The polynomial model (fit.cuh): four phases over all partitions, each its own kernel. Phases 1
// and 3 read the values (a warp per partition), phases 2 and 4 are a thread per partition. A map
// says where partition p's values are: one column (OneColumn), or the polynomial columns of a
// batch (BatchColumns; partitions of the batch's other columns are skipped).
struct OneColumn {
  const void* values;
  uint64_t n;
  const uint64_t* starts;
  uint32_t L;
  __device__ __forceinline__ bool get(uint64_t p, const void** v, uint64_t* a, uint32_t* N, uint32_t* slot) const {
    *v = values;
    *a = part_begin(starts, L, n, p);
    *N = (uint32_t)(part_begin(starts, L, n, p + 1) - *a);
    *slot = 0;
    return true;
  }
};

struct BatchColumns {
  const EncCol* cols;
  const uint64_t* part_base;
  uint32_t ncols;
  __device__ __forceinline__ bool get(uint64_t p, const void** v, uint64_t* a, uint32_t* N, uint32_t* slot) const {
    const uint32_t c = find_col(part_base, ncols, p);
    const EncCol col = cols[c];
    if (col.model != LECO_MODEL_POLY) return false;
    const uint64_t s = (p - part_base[c]) * (uint64_t)col.L;
    *v = col.values;
    *a = s;
    *N = (uint32_t)((s + col.L < col.n ? s + col.L : col.n) - s);
    *slot = c;
    return true;
  }
};

template <typename Map>
__global__ void __launch_bounds__(kFitBlock)
    k_poly_moments(const Map map, int dtype, uint64_t m, PolyMom* __restrict__ mom) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nw = (uint64_t)gridDim.x * kFitWarps;
  for (uint64_t p = (uint64_t)blockIdx.x * kFitWarps + (threadIdx.x >> 5); p < m; p += nw) {
    const void* v;
    uint64_t a;
    uint32_t N, slot;
    if (!map.get(p, &v, &a, &N, &slot)) continue;
    const PolyMom M = poly_moments_warp(v, dtype, a, N, lane);
    if (lane == 0) mom[p] = M;
  }
}

template <typename Map>
__global__ void k_poly_plan(const Map map, uint64_t m, const PolyMom* __restrict__ mom, PolyPlan* __restrict__ plan) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m; p += (uint64_t)gridDim.x * blockDim.x) {
    const void* v;
    uint64_t a;
    uint32_t N, slot;
    if (map.get(p, &v, &a, &N, &slot)) plan[p] = poly_plan(mom[p], N);
  }
}

template <typename Map>
__global__ void __launch_bounds__(kFitBlock)
    k_poly_ranges(const Map map, int dtype, uint64_t m, const PolyPlan* __restrict__ plan, PolyRange* __restrict__ rng) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t nw = (uint64_t)gridDim.x * kFitWarps;
  for (uint64_t p = (uint64_t)blockIdx.x * kFitWarps + (threadIdx.x >> 5); p < m; p += nw) {
    const void* v;
    uint64_t a;
    uint32_t N, slot;
    if (!map.get(p, &v, &a, &N, &slot)) continue;
    const PolyRange R = poly_ranges_warp(v, dtype, a, N, lane, plan + p);
    if (lane == 0) rng[p] = R;
  }
}

// the record (offset 0, set by the offset scan), stream bits, block and widest width of the choice
// (max_b[slot]: the column's)
template <typename Map>
__global__ void k_poly_choose(const Map map, uint64_t m, const PolyMom* __restrict__ mom,
                              const PolyPlan* __restrict__ plan, const PolyRange* __restrict__ rng,
                              Record* __restrict__ rec, uint64_t* __restrict__ lenbits, PolyCoef* __restrict__ pcoef,
                              uint32_t* __restrict__ max_b) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m; p += (uint64_t)gridDim.x * blockDim.x) {
    const void* v;
    uint64_t a;
    uint32_t N, slot;
    if (!map.get(p, &v, &a, &N, &slot)) continue;
    const FitChoice C = poly_choose(mom[p], plan[p], rng[p], N);
    Record r;
    r.start = a;
    if (C.kind >= 2) {
      r.theta0 = 0.0;
      r.theta1 = 0.0;
      r.word3 = make_w3(0, C.b, 0, 0) | kPolyFlag;
      pcoef[p] = C.pc;
      lenbits[p] = kPolyBlockBits + (uint64_t)N * C.b;
    } else {
      r.theta0 = C.R.theta0;
      r.theta1 = C.R.theta1;
      r.word3 = make_w3(0, C.R.b, C.R.s, 1);
      lenbits[p] = (uint64_t)N * C.R.b;
    }
    rec[p] = r;
    if (C.b) atomicMax(max_b + slot, C.b);
  }
}

// ------------------------------------------------------------------------------ exclusive scan

constexpr int kPrefixBlock = 256;
constexpr int kPrefixItems = 8;
constexpr uint64_t kPrefixTile = kPrefixBlock * kPrefixItems;

__device__ __forceinline__ uint64_t block_exclusive_scan(uint64_t v, uint64_t* warp_tot,
                                                         uint64_t* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint64_t inc = v;
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) warp_tot[wid] = inc;
  __syncthreads();
  if (wid == 0) {
    uint64_t t = lane < (kPrefixBlock / 32) ? warp_tot[lane] : 0;
    uint64_t ti = t;
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t u = __shfl_up_sync(0xffffffffu, ti, o);
      if (lane >= o) ti += u;
    }
    if (lane < (kPrefixBlock / 32)) warp_tot[lane] = ti - t;
    if (lane == (kPrefixBlock / 32) - 1) *total = ti;
  }
  __syncthreads();
  const uint64_t r = warp_tot[wid] + inc - v;
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kPrefixBlock)
    k_prefix_tiles(const uint64_t* __restrict__ in, uint64_t count, uint64_t* __restrict__ tile_sums) {
  const uint64_t base = (uint64_t)blockIdx.x * kPrefixTile;
  uint64_t s = 0;
  for (int k = 0; k < kPrefixItems; k++) {
    const uint64_t i = base + (uint64_t)k * kPrefixBlock + threadIdx.x;
    if (i < count) s += in[i];
  }
  s = warp_sum_u64(s);
  __shared__ uint64_t ws[kPrefixBlock / 32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t t = 0;
    for (int k = 0; k < kPrefixBlock / 32; k++) t += ws[k];
    tile_sums[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kPrefixBlock)
    k_prefix_top(uint64_t* __restrict__ tile_sums, uint64_t ntiles, uint64_t* __restrict__ total) {
  __shared__ uint64_t wt[kPrefixBlock / 32];
  __shared__ uint64_t tot;
  uint64_t carry = 0;
  for (uint64_t base = 0; base < ntiles; base += kPrefixBlock) {
    const uint64_t i = base + threadIdx.x;
    const uint64_t v = i < ntiles ? tile_sums[i] : 0;
    const uint64_t ex = block_exclusive_scan(v, wt, &tot);
    if (i < ntiles) tile_sums[i] = carry + ex;
    __syncthreads();
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(kPrefixBlock)
    k_prefix_apply(const uint64_t* __restrict__ in, uint64_t count,
                 const uint64_t* __restrict__ tile_prefix, uint64_t* __restrict__ out) {
  __shared__ uint64_t wt[kPrefixBlock / 32];
  __shared__ uint64_t tot;
  const uint64_t base = (uint64_t)blockIdx.x * kPrefixTile + (uint64_t)threadIdx.x * kPrefixItems;
  uint64_t v[kPrefixItems];
  uint64_t s = 0;
  for (int k = 0; k < kPrefixItems; k++) {
    const uint64_t i = base + k;
    v[k] = i < count ? in[i] : 0;
    s += v[k];
  }
  uint64_t run = block_exclusive_scan(s, wt, &tot) + tile_prefix[blockIdx.x];
  for (int k = 0; k < kPrefixItems; k++) {
    const uint64_t i = base + k;
    if (i < count) out[i] = run;
    run += v[k];
  }
}

// Offsets of a column of up to kOneCtaParts partitions in one launch: each thread sums a run of lengths, the
// CTA scans the sums, then each thread writes its run. Four launches of the general scan took 11 us of a
// 100K-value encode (98 partitions) besides their launches, this 4 us.
constexpr int kOneCtaBlock = 1024;
constexpr uint64_t kOneCtaParts = 8 * kOneCtaBlock;  // at 20,000 partitions the general scan is as fast

__global__ void __launch_bounds__(kOneCtaBlock)
    k_offsets_one(Record* __restrict__ rec, const uint64_t* __restrict__ lenbits, uint32_t m, uint64_t* __restrict__ total) {
  __shared__ uint64_t ws[32];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const uint32_t per = (m + kOneCtaBlock - 1) / kOneCtaBlock, p0 = min(t * per, m), p1 = min(p0 + per, m);
  uint64_t sum = 0;
#pragma unroll 8
  for (uint32_t p = p0; p < p1; p++) sum += lenbits[p];
  uint64_t inc = sum;
  for (uint32_t o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) ws[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint64_t w = ws[lane];
    uint64_t wi = w;
    for (uint32_t o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    ws[lane] = wi - w;
    if (lane == 31) *total = wi;
  }
  __syncthreads();
  uint64_t off = ws[warp] + inc - sum;
#pragma unroll 8
  for (uint32_t p = p0; p < p1; p++) {
    rec[p].word3 = (rec[p].word3 & ~kOffMask) | (off & kOffMask);
    off += lenbits[p];
  }
}

__global__ void k_set_offsets(Record* __restrict__ rec, const uint64_t* __restrict__ off, uint64_t m) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < m;
       p += (uint64_t)gridDim.x * blockDim.x)
    rec[p].word3 = (rec[p].word3 & ~kOffMask) | (off[p] & kOffMask);
}

// ------------------------------------------------------------------------------ decode table

// Verify the exact flag of each record and derive the grid integers; a record that does not pass
// keeps the binary64 path (the definition), so a foreign or damaged header can never decode
// differently from the prediction it states.
__device__ Aux aux_of(const Record& r, uint64_t N) {
  {
    Aux a;
    a.start = r.start;
    a.A = 0;
    a.B = 0;
    bool ok = w3_exact(r.word3) && N >= 1 && N <= kMaxPartLen;
    const int s = w3_s(r.word3);
    ok = ok && s >= -11 && s <= 52;
    if (ok) {
      const double fa = r.theta0 * pow2(s), fb = r.theta1 * pow2(s);  // exact power-of-two scale
      const double lim53 = 9007199254740992.0;                        // 2^53
      ok = fa == floor(fa) && fb == floor(fb) && fabs(fa) < lim53 && fabs(fb) < lim53;
      if (ok) {
        const int64_t A = (int64_t)fa, B = (int64_t)fb;
        const i128 f0 = A, f1 = (i128)A + (i128)B * (i128)(N - 1);
        const i128 bx = (i128)B * (i128)(N - 1);
        const i128 l53 = (i128)1 << 53;
        ok = f0 < l53 && f0 > -l53 && f1 < l53 && f1 > -l53 && bx < l53 && bx > -l53;
        if (ok && s < 0) {  // scaled values must stay inside int64 (no saturation)
          const i128 g = (i128)1 << (-s);
          const i128 l63 = (i128)1 << 63;
          ok = f0 * g < l63 && f0 * g >= -l63 && f1 * g < l63 && f1 * g >= -l63;
          if (ok) {
            a.A = (int64_t)(f0 * g);
            a.B = (int64_t)((i128)B * g);
          }
        } else if (ok) {
          a.A = A;
          a.B = B;
        }
      }
    }
    a.word3 = ok ? r.word3 : (r.word3 & ~(1ull << 62));
    return a;
  }
}

// decode-table entry and polynomial table row of a polynomial partition (block pc, N values)
__device__ Aux poly_entry(const Record& r, const PolyCoef& pc, uint32_t N, PolyAux* row) {
  int32_t sj[3], S = 0;
  for (int j = 0; j < 3; j++) {
    sj[j] = (int32_t)((pc.E >> (8 * j)) & 0xFF);
    S = max(S, sj[j]);
  }
  *row = poly_aux_from(pc.K, sj, S, N);
  Aux a;
  a.A = pc.T;
  a.B = 0;
  a.start = r.start;
  a.word3 = make_w3(w3_off(r.word3) + kPolyBlockBits, w3_b(r.word3), S, 0) | kPolyFlag;
  return a;
}

// first stream bit of a partition: its residuals, or the block ahead of them for a polynomial one
__device__ __forceinline__ uint64_t part_first_bit(const Aux& a) {
  return w3_off(a.word3) - (w3_poly(a.word3) ? kPolyBlockBits : 0);
}

// zeroes the words that packing OR-s into at the start of one partition: the word of its first bit and
// those of a coefficient block
__device__ __forceinline__ void zero_bound(const Aux& a, uint64_t* __restrict__ words) {
  const uint64_t w = part_first_bit(a) >> 6, e = w3_off(a.word3) >> 6;
  for (uint64_t k = w; k <= e; k++) words[k] = 0;
}

__device__ __forceinline__ Aux entry_of(const Record& r, const PolyCoef* __restrict__ pcoef, PolyAux* __restrict__ poly,
                                        uint64_t p, uint64_t N) {
  return w3_poly(r.word3) && pcoef && poly ? poly_entry(r, pcoef[p], (uint32_t)N, poly + p) : aux_of(r, N);
}

// The decode table and, for a stream about to be packed (words), zeroes in the words that packing OR-s
// into: each word holding a partition's first bit (and its block), and the words from the end of the stream
// on (the tail word and the zero padding). Every other word lies inside one partition's bit range and is
// written whole. Clears the column's status word.
__global__ void k_build_aux(const Record* __restrict__ rec, const PolyCoef* __restrict__ pcoef, uint64_t m,
                            uint64_t n, Aux* __restrict__ aux, PolyAux* __restrict__ poly, uint64_t total_bits,
                            uint64_t nwords, uint64_t* __restrict__ words, uint32_t* __restrict__ status) {
  const uint64_t tail = total_bits >> 6;
  const uint64_t count = m + (words && nwords > tail ? nwords - tail : 0);
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
    if (i == 0 && status) *status = 0;
    if (i >= m) {
      words[tail + (i - m)] = 0;
      continue;
    }
    const Record r = rec[i];
    const uint64_t e = i + 1 < m ? rec[i + 1].start : n;
    const Aux a = entry_of(r, pcoef, poly, i, e > r.start ? e - r.start : 0);
    aux[i] = a;
    if (words) zero_bound(a, words);
  }
}

// ------------------------------------------------------------------------------ packing
//
// A warp packs a window of consecutive positions, whatever partitions it touches: no barrier, no warp
// waits for another, and partitions of any length take the same path; the windows shrink until a small
// column fills the GPU. The piece of a partition inside a window owns the 32-bit words whose last bit
// lies in it (at the partition's end, its last word too), so each word inside a partition is written
// once, by one warp, with a few values before the piece read again. Words that hold a partition
// boundary (or the end of the stream) were zeroed beforehand and are OR-ed into.
//
// The values' residuals go to a shared tile of 32 rows of K = 8, 16 or 32 consecutive values; lane r takes
// row r into registers, strings its bits together from their place in the piece's words on (no division,
// two values at a time up to 16 bits), passes the open last word to the next lane and leaves the others in
// the tile, from where they go out coalesced. Widths above 32 bits take 64-bit entries and rows of 8 (20M values of 63
// bits in partitions of 4096 116 -> 75 us, of 40 bits 88 -> 63 us, against each word assembled from the fields it
// holds); pieces of up to 128 such values, wide polynomial and binary64 partitions still assemble words (pack_words).
// The former packer staged a partition, or a run of short ones, per CTA by a bulk copy, three to seven
// CTAs per SM each waiting for its own, and recomputed every field of partitions beyond 4096 values
// from memory. Bound: memory and the latency of a piece's chain (64 registers hold 32 warps per SM; 48, 40
// or 80 registers were slower). Measured, former -> this: 200M sorted normal uint64 in partitions of 4096
// 431 -> 351 us (5.7 TB/s), 250M 32-bit timestamps in variable partitions 1295 -> 531 us, 100M piecewise
// values 2.39 -> 0.9 ms, 96 columns of 200M values in partitions of 256 .. 4096 492 -> 431 us, 20M 32-bit
// values in partitions of 1000 83 -> 44 us.
constexpr int kPackBlock = 256;
constexpr int kPackWarps = kPackBlock / 32;
constexpr int kPackCtas = 4;  // CTAs per SM the registers are held for
constexpr int kChunkLoads = 9;
constexpr uint32_t kChunkVals = 32 * kChunkLoads;
constexpr uint32_t kPackPiece = 1024;   // values packed at a time
constexpr uint32_t kPackWindow = 4096;  // positions per warp of a large column
constexpr uint32_t kPackTile = 32 * 33;  // 32-bit entries of a warp's tile
static_assert(kPackTile * 4 >= kChunkVals * 8, "a chunk's 64-bit residuals fit the tile");

template <bool POLY>
__device__ __forceinline__ uint64_t residual_at(const Record* __restrict__ rec, const PolyAux* __restrict__ poly,
                                                const Aux& a, uint64_t p, uint32_t x, uint64_t v) {
  const int64_t pred = POLY ? predict_aux(a, rec, poly, p, x) : predict_aux_line(a, rec, p, x);
  return zz_encode((int64_t)(v - (uint64_t)pred));
}

// a partition being packed
template <typename T>
struct PackPart {
  const T* v;            // its first value
  uint32_t N, b, magic;  // values, width, ceil(2^32 / b) for b > 1: floor(r / b) as a high product, exact
                         // for r < 2^26 (a chunk or piece has at most 2^16 bits)
  uint32_t lead;         // bit of out[0] where its residuals begin
  uint32_t* out;
  uint64_t A, B;
  uint32_t sh;
  uint64_t p;
  __device__ __forceinline__ uint32_t div_b(uint32_t r) const { return b > 1 ? __umulhi(r, magic) : r; }
  // word w lies inside the partition's bits
  __device__ __forceinline__ bool whole(uint32_t w) const {
    return (w > 0 || lead == 0) && 32u * w + 32u <= lead + N * b;
  }
  __device__ __forceinline__ void put(uint32_t w, uint32_t x) const {
    if (whole(w))
      out[w] = x;
    else
      atomicOr(out + w, x);
  }
};

// words [w0, w1) of a partition, each assembled from the fields it holds, a chunk of at most
// kChunkVals values at a time
template <typename T, bool POLY>
__device__ __forceinline__ void pack_words(const PackPart<T>& q, const Aux& a, const Record* __restrict__ rec,
                                           const PolyAux* __restrict__ poly, uint32_t w0, uint32_t w1, uint64_t* zs,
                                           uint32_t lane) {
  const uint32_t b = q.b;
  const uint32_t most = ((kChunkVals - 2) * b) >> 5;  // words that at most kChunkVals fields overlap
  const bool line = w3_exact(a.word3) != 0, pl = POLY && w3_poly(a.word3) != 0;
  for (uint32_t w = w0; w < w1; w += most) {
    const uint32_t we = min(w + most, w1);
    const int32_t rb = (int32_t)(32u * w) - (int32_t)q.lead;
    const uint32_t x_lo = rb > 0 ? (uint32_t)rb / b : 0u;
    const int32_t rl = rb - (int32_t)(x_lo * b);  // below 0 where the partition begins inside the word
    const uint32_t x_hi = min(q.N, x_lo + q.div_b((uint32_t)(rl + (int32_t)(32u * (we - w) + b - 1u))));
    T val[kChunkLoads];
#pragma unroll
    for (int k = 0; k < kChunkLoads; k++) {
      const uint32_t x = x_lo + lane + 32u * k;
      val[k] = x < x_hi ? __ldg(q.v + x) : (T)0;
    }
    if (line) {
      uint64_t F = q.A + q.B * (x_lo + lane);
#pragma unroll
      for (int k = 0; k < kChunkLoads; k++, F += q.B * 32u)
        zs[lane + 32 * k] = zz_encode((int64_t)((uint64_t)val[k] - (uint64_t)((int64_t)F >> q.sh)));
    } else if (pl) {
      PolySteps Fd = poly_steps(poly[q.p], x_lo + lane, 32, 64u - ((uint32_t)w3_s(a.word3) & 63u));
#pragma unroll
      for (int k = 0; k < kChunkLoads; k++) {
        zs[lane + 32 * k] = zz_encode((int64_t)((uint64_t)val[k] - ((uint64_t)a.A + (uint64_t)(Fd.F >> 64))));
        poly_step(Fd);
      }
    } else {
#pragma unroll 1
      for (int k = 0; k < kChunkLoads; k++) {
        const uint32_t x = x_lo + lane + 32u * k;
        if (x < x_hi) zs[lane + 32 * k] = residual_at<POLY>(rec, poly, a, q.p, x, (uint64_t)__ldg(q.v + x));
      }
    }
    __syncwarp();
    const uint32_t V = x_hi - x_lo;
    for (uint32_t j = lane; j < we - w; j += 32) {
      const int32_t r = rl + (int32_t)(32u * j);
      uint32_t x = r > 0 ? q.div_b((uint32_t)r) : 0u;
      uint32_t acc = 0;
      for (int32_t f = (int32_t)(x * b) - r; f < 32 && x < V; f += (int32_t)b, x++) {
        const uint64_t z = zs[x];
        acc |= f >= 0 ? (uint32_t)z << f : (uint32_t)(z >> (-f));
      }
      q.put(w + j, acc);
    }
    __syncwarp();
  }
}

// values [x0, x0 + V) of a partition of width b <= 32 on a line (or, PL, a polynomial), V <= 32 K, K b >= 32:
// lane r packs the K consecutive values of row r. WIDE: widths above 32 bits, K = 8; a value goes in as its low 32
// bits and the rest.
template <int K, typename T, bool PL, bool WIDE = false>
__device__ __forceinline__ void pack_rows(const PackPart<T>& q, const Aux& a, const PolyAux* __restrict__ poly,
                                          uint32_t x0, uint32_t V, uint32_t* tile, uint32_t lane) {
  const uint32_t b = q.b;
  PolySteps Fd;
  if (PL) Fd = poly_steps(poly[q.p], x0 + lane, 32, 64u - ((uint32_t)w3_s(a.word3) & 63u));
  const T* v = q.v + x0 + lane;
  // the lane loads values lane + 32 k for k < mine (x < V); steps past them leave bits past the piece
  const int mine = V > lane ? (int)((V - lane + 31u) >> 5) : 0;
  uint64_t F = q.A + q.B * (x0 + lane);
  const uint64_t dF = q.B * 32u;
  T val[2][8];
#pragma unroll
  for (int u = 0; u < 8; u++) val[0][u] = u < mine ? __ldg(v + 32 * u) : (T)0;
  // a width of at most 32 bits: the zigzag code is 32 bits of the residual and its sign
  auto zz32 = [](uint64_t r) { return ((uint32_t)r << 1) ^ (uint32_t)((int32_t)(r >> 32) >> 31); };
  // the bits before the piece in its first word, from the values that hold them
  const uint32_t bit = q.lead + x0 * b, w0 = bit >> 5, o = bit & 31u;
  uint32_t prev = 0;
  if (x0 && o) {
    uint32_t c = 0;
    if (lane * b < o && lane < x0) {
      const uint32_t x = x0 - 1u - lane;
      const uint64_t pred = PL ? (uint64_t)predict_aux(a, nullptr, poly, q.p, x) : (uint64_t)((int64_t)(q.A + q.B * x) >> q.sh);
      const uint64_t r = (uint64_t)__ldg(q.v + x) - pred;
      const int32_t s = (int32_t)o - (int32_t)((lane + 1u) * b);
      if (WIDE)
        c = (uint32_t)(zz_encode((int64_t)r) >> (-s));  // o < 32 < b
      else
        c = s >= 0 ? zz32(r) << s : zz32(r) >> (-s);
    }
    prev = __reduce_or_sync(0xffffffffu, c);
  }
  using Z = typename std::conditional<WIDE, uint64_t, uint32_t>::type;
  Z* zs = reinterpret_cast<Z*>(tile);
  Z* put = zs + lane + (K == 32 ? 0u : lane / (uint32_t)K);
#pragma unroll
  for (int k = 0; k < K; k += 8) {
    const int cur = (k >> 3) & 1;
    if (k + 8 < K) {
#pragma unroll
      for (int u = 0; u < 8; u++) val[cur ^ 1][u] = k + 8 + u < mine ? __ldg(v + 32 * (k + 8 + u)) : (T)0;
    }
#pragma unroll
    for (int u = 0; u < 8; u++) {
      uint64_t pred;
      if (PL) {
        pred = (uint64_t)a.A + (uint64_t)(Fd.F >> 64);
        poly_step(Fd);
      } else {
        pred = (uint64_t)((int64_t)F >> q.sh);
        F += dF;
      }
      const uint64_t r = (uint64_t)val[cur][u] - pred;
      put[(32 + 32 / K) * (k + u)] = WIDE ? (Z)zz_encode((int64_t)r) : (Z)zz32(r);  // value x at x + x / K
    }
  }
  __syncwarp();
  // The row's bits begin at bit `at` of the piece's words; its first word and the open last one are put
  // together with the neighbours'. Rows of 32 values begin at the same bit of a word in every lane, b words
  // apart: `fill` and the branches on it are uniform, and the words replace the row's residuals in place
  // (word k is complete after more than k values). Shorter rows go through registers to the tile as one
  // run of words, every 33rd free so that rows a power of two apart use different banks.
  const uint32_t at = o + lane * (uint32_t)K * b, wf = at >> 5;
  uint32_t first = 0, open = 0;
  if (K == 32) {
    uint32_t* row = tile + lane * 33u;
    uint32_t fill = o, done = 0, acc = 0;
    auto emit = [&](uint32_t x, uint32_t width) {  // x < 2^width, or bits past the piece
      const uint64_t t = (uint64_t)x * (1u << fill) + acc;
      acc = (uint32_t)t;
      fill += width;
      if (fill >= 32u) {
        row[done++] = acc;
        acc = (uint32_t)(t >> 32);
        fill -= 32u;
      }
    };
    if (b <= 16) {
      const uint32_t pw = 1u << b;
#pragma unroll 8
      for (int i = 0; i < K; i += 2) emit(row[i] + row[i + 1] * pw, 2u * b);
    } else {
#pragma unroll 8
      for (int i = 0; i < K; i++) emit(row[i], b);
    }
    open = acc;
  } else {
    Z z[K];
#pragma unroll
    for (int i = 0; i < K; i++) z[i] = zs[lane * (K + 1) + i];
    __syncwarp();
    uint32_t w = wf, fill = at & 31u, acc = 0;
    auto emit = [&](uint32_t x, uint32_t width) {
      const uint64_t t = (uint64_t)x * (1u << fill) + acc;
      const bool full = fill + width >= 32u;
      if (full && w != wf) tile[w + (w >> 5)] = (uint32_t)t;
      if (full && w == wf) first = (uint32_t)t;
      acc = full ? (uint32_t)(t >> 32) : (uint32_t)t;
      fill = (fill + width) & 31u;
      w += full ? 1u : 0u;
    };
    if (WIDE) {
#pragma unroll
      for (int i = 0; i < K; i++) {
        emit((uint32_t)z[i], 32u);
        emit((uint32_t)((uint64_t)z[i] >> 32), b - 32u);
      }
    } else if (b <= 16) {
      const uint32_t pw = 1u << b;
#pragma unroll
      for (int i = 0; i < K; i += 2) emit((uint32_t)z[i] + (uint32_t)z[i + 1] * pw, 2u * b);
    } else {
#pragma unroll
      for (int i = 0; i < K; i++) emit((uint32_t)z[i], b);
    }
    open = acc;
  }
  uint32_t below = __shfl_up_sync(0xffffffffu, open, 1);
  if (lane == 0) below = prev;
  if (K == 32)
    tile[lane * 33u] |= below;
  else
    tile[wf + (wf >> 5)] = first | below;
  const uint32_t past = (at + (uint32_t)K * b) >> 5;  // the open word
  const uint32_t tail = __shfl_sync(0xffffffffu, open, 31), wtail = __shfl_sync(0xffffffffu, past, 31);
  __syncwarp();
  auto word = [&](uint32_t j) -> uint32_t {
    if (j == wtail) return tail;
    if (K != 32) return tile[j + (j >> 5)];
    const uint32_t r = q.div_b(j);
    return tile[r * 33u + (j - r * b)];
  };
  const uint32_t end = o + V * b;
  const bool last = x0 + V == q.N;
  // words that lie inside the partition's bits are stored, its first and last one OR-ed into
  const uint32_t j0 = q.lead && w0 == 0 ? 1u : 0u, j1 = end >> 5;
  uint32_t* out = q.out + w0;
  for (uint32_t j = j0 + lane; j < j1; j += 32) out[j] = word(j);
  if (lane == 0 && j0) {
    const uint32_t keep = j1 == 0 ? (1u << (end & 31u)) - 1u : ~0u;
    if (j1 || last) atomicOr(out, word(0) & keep);
  }
  if (lane == 1 && last && (end & 31u) && j1 >= j0) atomicOr(out + j1, word(j1) & ((1u << (end & 31u)) - 1u));
  __syncwarp();
}

// values [xa, xb) of a partition of N values (its first value at v[0], entry a, index p)
template <typename T, bool POLY, bool WIDE>
__device__ __forceinline__ void pack_piece(const T* __restrict__ v, uint32_t N, uint32_t xa, uint32_t xb, const Aux& a,
                                           const Record* __restrict__ rec, const PolyAux* __restrict__ poly, uint64_t p,
                                           uint32_t* __restrict__ words, uint64_t* zbuf, uint32_t lane) {
  PackPart<T> q;
  q.b = w3_b(a.word3);
  if (q.b == 0) return;
  q.v = v;
  q.N = N;
  q.magic = 0xFFFFFFFFu / q.b + 1u;  // b = 1 takes no product
  const uint64_t off = w3_off(a.word3);
  q.lead = (uint32_t)off & 31u;
  q.out = words + (off >> 5);
  q.A = (uint64_t)a.A;
  q.B = (uint64_t)a.B;
  const int32_t sr = w3_s(a.word3);
  q.sh = sr > 0 ? (uint32_t)sr & 63u : 0u;
  q.p = p;
  const bool line = w3_exact(a.word3) != 0, pl = POLY && w3_poly(a.word3) != 0;
  uint32_t* tile = reinterpret_cast<uint32_t*>(zbuf);
  if (WIDE && q.b > 32 && line && xb - xa > 128) {  // shorter pieces leave most of the 32 rows empty
    for (uint32_t x = xa; x < xb; x += 256) pack_rows<8, T, false, true>(q, a, poly, x, min(256u, xb - x), tile, lane);
    return;
  }
  if (q.b <= 32 && (line || pl)) {
    for (uint32_t x = xa; x < xb; x += kPackPiece) {
      const uint32_t V = min(kPackPiece, xb - x);
      if (pl)
        pack_rows<32, T, true>(q, a, poly, x, V, tile, lane);
      else if (V <= 256 && q.b >= 4)
        pack_rows<8, T, false>(q, a, poly, x, V, tile, lane);
      else if (V <= 512 && q.b >= 2)
        pack_rows<16, T, false>(q, a, poly, x, V, tile, lane);
      else
        pack_rows<32, T, false>(q, a, poly, x, V, tile, lane);
    }
    return;
  }
  const uint32_t w0 = (q.lead + xa * q.b) >> 5;
  const uint32_t w1 = xb == N ? (q.lead + N * q.b + 31u) >> 5 : (q.lead + xb * q.b) >> 5;
  pack_words<T, POLY>(q, a, rec, poly, w0, w1, zbuf, lane);
}

// the coefficient block of a polynomial partition, ten 32-bit words at the bit before its residuals:
// OR-ed, as are the words' other bits (k_build_aux zeroed them)
__device__ __forceinline__ void pack_block(const PolyCoef& pc, uint64_t off0, uint32_t* __restrict__ words, uint32_t lane) {
  if (lane >= 10) return;
  const uint32_t q = lane >> 1;
  const uint64_t f = q == 0 ? (uint64_t)pc.T : q == 4 ? pc.E : (uint64_t)(q == 1 ? pc.K[0] : q == 2 ? pc.K[1] : pc.K[2]);
  const uint32_t h = (lane & 1u) ? (uint32_t)(f >> 32) : (uint32_t)f;
  const uint64_t at = off0 + 32ull * lane;
  const uint32_t o = (uint32_t)at & 31u;
  uint32_t* w = words + (at >> 5);
  atomicOr(w, h << o);
  if (o) atomicOr(w + 1, h >> (32u - o));
}

// A whole partition on a line by one lane: its bits strung together from the place of its first one, whole words
// stored, the shared ones at its ends OR-ed into. For short ones (lane_part_of, and at most kLaneBits bits: beyond
// them the words of 32 lanes are too far apart); a warp spends about 600 instructions on each.
template <typename T>
__device__ __forceinline__ void pack_lane(const T* __restrict__ v, uint32_t N, const Aux& a, uint32_t* __restrict__ words) {
  const uint32_t b = w3_b(a.word3);
  if (b == 0) return;
  const uint64_t off = w3_off(a.word3);
  const int32_t sr = w3_s(a.word3);
  const uint32_t sh = sr > 0 ? (uint32_t)sr & 63u : 0u;
  uint32_t* out = words + (off >> 5);
  uint32_t fill = (uint32_t)off & 31u, acc = 0;
  bool shared = fill != 0;  // the first word holds another partition's bits too
  auto emit = [&](uint32_t x, uint32_t width) {
    const uint64_t t = ((uint64_t)x << fill) | acc;
    acc = (uint32_t)t;
    fill += width;
    if (fill >= 32u) {
      if (shared)
        atomicOr(out, acc);
      else
        *out = acc;
      shared = false;
      out++;
      acc = (uint32_t)(t >> 32);
      fill -= 32u;
    }
  };
  uint64_t F = (uint64_t)a.A;
  for (uint32_t x = 0; x < N; x += 4) {
    T val[4];
#pragma unroll
    for (int k = 0; k < 4; k++) val[k] = x + k < N ? __ldg(v + x + k) : (T)0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
      if (x + k < N) {
        const uint64_t z = zz_encode((int64_t)((uint64_t)val[k] - (uint64_t)((int64_t)F >> sh)));
        F += (uint64_t)a.B;
        emit((uint32_t)z, min(b, 32u));
        if (b > 32) emit((uint32_t)(z >> 32), b - 32u);
      }
    }
  }
  if (fill) atomicOr(out, acc);
}

// positions [pos, end) of a column, partition p holding pos
template <typename T, bool POLY, bool SHORT, bool WIDE>
__device__ __forceinline__ void pack_window(const T* __restrict__ values, uint64_t n, uint64_t m, uint64_t pos,
                                            uint64_t end, uint64_t p, const Record* __restrict__ rec,
                                            const Aux* __restrict__ aux, const PolyCoef* __restrict__ pcoef,
                                            const PolyAux* __restrict__ poly, uint32_t* __restrict__ words,
                                            uint64_t* zbuf, uint32_t lane, uint32_t lane_part) {
  // the lanes fetch 32 entries at a time (one memory round trip for a run of short partitions)
  while (pos < end) {
    Aux mine;
    mine.A = mine.B = 0;
    mine.word3 = 0;
    mine.start = n;
    if (p + lane < m) mine = aux[p + lane];
    uint32_t lanes = 0;  // short partitions that lie inside the window whole: a lane each, all at once
    if (SHORT) {
      const uint64_t next = __shfl_down_sync(0xffffffffu, mine.start, 1);
      lanes = __ballot_sync(0xffffffffu, lane < 31 && mine.start >= pos && mine.start < next && next <= end &&
                                             next - mine.start <= lane_part && w3_exact(mine.word3) &&
                                             (next - mine.start) * w3_b(mine.word3) <= kLaneBits);
      if (__popc(lanes) < 2)
        lanes = 0;
      else if ((lanes >> lane) & 1u)
        pack_lane(values + mine.start, (uint32_t)(next - mine.start), mine, words);
    }
    for (uint32_t k = 0; k < 31 && pos < end; k++, p++) {
      if (SHORT && ((lanes >> k) & 1u)) {  // on to the next partition that is left
        const uint32_t run = (uint32_t)__ffs((int)~(lanes >> k)) - 1u;
        pos = __shfl_sync(0xffffffffu, mine.start, k + run);
        k += run - 1u;
        p += run - 1u;
        continue;
      }
      Aux a;
      a.A = __shfl_sync(0xffffffffu, mine.A, k);
      a.B = __shfl_sync(0xffffffffu, mine.B, k);
      a.start = __shfl_sync(0xffffffffu, mine.start, k);
      a.word3 = __shfl_sync(0xffffffffu, mine.word3, k);
      const uint64_t e = __shfl_sync(0xffffffffu, mine.start, k + 1);
      const uint32_t xa = (uint32_t)(pos - a.start);
      if (POLY && xa == 0 && w3_poly(a.word3)) pack_block(pcoef[p], w3_off(a.word3) - kPolyBlockBits, words, lane);
      pack_piece<T, POLY, WIDE>(values + a.start, (uint32_t)(e - a.start), xa, (uint32_t)(min(e, end) - a.start), a, rec, poly,
                          p, words, zbuf, lane);
      pos = e;
    }
  }
}

// WIDE: some partition of the column is wider than 32 bits (a kernel of its own, since the others would be 2 - 4 %
// slower beside those rows). L: the fixed partition length, or 0: partitions of any lengths, found through the scan
// tiles. Every `period`
// positions hold `per` windows, the last one shorter where they do not divide it.
template <typename T, bool POLY, bool SHORT, bool WIDE>
__global__ void __launch_bounds__(kPackBlock, POLY ? 2 : kPackCtas)
    k_pack(const T* __restrict__ values, uint64_t n, uint64_t m, uint32_t L, uint32_t window, uint32_t period,
           uint32_t per, const TileDesc* __restrict__ tiles, const Record* __restrict__ rec,
           const Aux* __restrict__ aux, const PolyCoef* __restrict__ pcoef, const PolyAux* __restrict__ poly,
           uint32_t* __restrict__ words, uint32_t lane_part) {
  __shared__ uint64_t zbuf[kPackWarps][kPackTile / 2];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint64_t nwin = (n + period - 1) / period * per, nw = (uint64_t)gridDim.x * kPackWarps;
  for (uint64_t k = (uint64_t)blockIdx.x * kPackWarps + wid; k < nwin; k += nw) {
    const uint64_t q = per == 1 ? k : k / per, from = q * period, pos = from + (k - q * per) * window;
    const uint64_t end = min(min(pos + window, from + period), n);
    if (pos >= end) continue;  // past the last partition's end
    uint64_t p;
    if (L) {
      p = pos / L;
    } else {
      const TileDesc* d = tiles + pos / kScanTile;
      p = d->p0;
      uint64_t hi = p + d->np;
      while (hi - p > 1) {
        const uint64_t mid = (p + hi) >> 1;
        if (aux[mid].start <= pos)
          p = mid;
        else
          hi = mid;
      }
    }
    pack_window<T, POLY, SHORT, WIDE>(values, n, m, pos, end, p, rec, aux, pcoef, poly, words, zbuf[wid], lane,
                                  lane_part);
  }
}

// ------------------------------------------------------------------------------ batched encode

// The partitions of every column (a partition's column from the partition-column table; the polynomial
// columns' are fitted by the polynomial phases), in groups of eight per pair of warps: a tile of eight lanes each
// when all are short, else both warps on one after another, as k_fit_pairs. PARTS: the groups of long partitions
// are dealt out in `parts` parts (fit_parts), where whole groups would leave pairs without work or some with far
// more than others; a column of 5M values in partitions of 4096 kept 153 of the GPU's 1824 pairs busy.
// MID: no partition is longer than kFitMidVals; sixteen lanes each, four at a time, where some are above kFitTileVals.
// A kernel of its own: beside the long ones' path these tiles cost it more in registers (84 -> 96 us for 50M values in
// partitions of 4096).
// This kernel's time, whole groups of long partitions -> parts: that column 47 -> 12 us, 20 columns of 8M values in
// all in partitions of 4096 53 -> 20 us, 60 columns of 50M values in partitions of 256, 1024 and 4096 231 -> 173 us.
// Both warps on one after another -> tiles of sixteen: 20 columns of 20M values in partitions of 600 105 -> 49 us (a
// warp each, formerly: 93), of 100M 32-bit values in partitions of 1000 246 -> 145 us.
constexpr uint32_t kFitTileVals = 512, kFitMidVals = 1024;

template <typename T, bool PARTS, bool MID>
__global__ void __launch_bounds__(kFitBlock, kPairCtas)
    k_fit_multi(const EncCol* __restrict__ cols, const uint64_t* __restrict__ part_base,
                const uint32_t* __restrict__ part_col, uint64_t P, uint32_t parts, Record* __restrict__ rec,
                uint64_t* __restrict__ lenbits, uint32_t* __restrict__ max_b) {
  __shared__ FitShared sm[kFitPairs];
  const uint32_t g = threadIdx.x >> 6, rank = threadIdx.x & 63u, lane = threadIdx.x & 31u;
  const uint64_t ng = (uint64_t)gridDim.x * kFitPairs, groups = (P + 7) / 8;
  const int per = PARTS ? 8 / (int)parts : 8;
  for (uint64_t t = (uint64_t)blockIdx.x * kFitPairs + g; t < (PARTS ? groups * parts : groups); t += ng) {
    // first parts of all groups, then the second ones: whole groups of short partitions go with the first
    const uint64_t part = PARTS ? t / groups : 0, p0 = (t - part * groups) * 8;
    const int k0 = (int)part * per;
    // lane k (and k + 8, + 16, + 24) of both warps: partition p0 + k
    const uint64_t p = p0 + (lane & 7u);
    uint64_t a = 0;
    uint32_t N = 0, c = 0;
    int model = LECO_MODEL_CONSTANT;
    const T* v = nullptr;
    if (p < P) {
      c = part_col[p];
      const EncCol col = cols[c];
      model = col.model;
      a = (p - part_base[c]) * (uint64_t)col.L;
      if (model != LECO_MODEL_POLY) N = (uint32_t)((a + col.L < col.n ? a + col.L : col.n) - a);
      v = static_cast<const T*>(col.values) + a;
    }
    // partitions from, from + 1, ... of the group, a tile of lanes each
    auto tiles = [&](auto width, int from) {
      constexpr int TILE = decltype(width)::value;
      const int k = from + (int)rank / TILE;
      const uint32_t n = __shfl_sync(0xffffffffu, N, k);
      const T* vk = reinterpret_cast<const T*>(__shfl_sync(0xffffffffu, (unsigned long long)v, k));
      const FitResult R = fit_tile<TILE>(vk, n, __shfl_sync(0xffffffffu, model, k), rank % TILE);
      const uint64_t ak = __shfl_sync(0xffffffffu, a, k);
      const uint32_t ck = __shfl_sync(0xffffffffu, c, k);
      if (rank % TILE == 0 && n) put_fit(R, ak, n, p0 + (uint32_t)k, rec, lenbits, max_b + ck);
    };
    if (__all_sync(0xffffffffu, N <= kFitTileVals)) {
      if (k0 == 0) tiles(std::integral_constant<int, 8>(), 0);
      continue;
    }
    if constexpr (MID) {
      for (int k = k0; k < k0 + per; k += 4) tiles(std::integral_constant<int, 16>(), k);
      continue;
    }
    for (int k = k0; k < k0 + per; k++) {
      const uint32_t n = __shfl_sync(0xffffffffu, N, k);
      if (n == 0) continue;
      const T* vk = reinterpret_cast<const T*>(__shfl_sync(0xffffffffu, (unsigned long long)v, k));
      const FitResult R = fit_range<64>(vk, sizeof(T) == 4 ? LECO_U32 : LECO_U64, 0, n,
                                        __shfl_sync(0xffffffffu, model, k), rank, &sm[g], 1 + (int)g);
      if (rank == (uint32_t)k) put_fit(R, a, N, p, rec, lenbits, max_b + c);
    }
  }
}

// column-relative offsets from the global exclusive scan, and each column's total bits
__global__ void k_set_offsets_multi(Record* __restrict__ rec, const uint64_t* __restrict__ off,
                                    const uint64_t* __restrict__ lenbits, const uint64_t* __restrict__ part_base,
                                    const uint32_t* __restrict__ part_col, uint64_t P,
                                    uint64_t* __restrict__ col_bits) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < P;
       p += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t c = part_col[p];
    const uint64_t base = off[part_base[c]];
    rec[p].word3 = (rec[p].word3 & ~kOffMask) | ((off[p] - base) & kOffMask);
    if (p + 1 == part_base[c + 1]) col_bits[c] = off[p] + lenbits[p] - base;
  }
}

// k_build_aux for every column: a thread per partition, then each column's tail words
__global__ void k_aux_multi(const Record* __restrict__ rec, const PolyCoef* __restrict__ pcoef,
                            const EncCol* __restrict__ cols, const uint64_t* __restrict__ part_base,
                            const uint32_t* __restrict__ part_col, const uint64_t* __restrict__ word_base,
                            const uint64_t* __restrict__ col_bits, uint32_t ncols, uint64_t P, Aux* __restrict__ aux,
                            PolyAux* __restrict__ poly, uint64_t* __restrict__ words) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < P; p += stride) {
    const uint32_t c = part_col[p];
    const Record r = rec[p];
    const uint64_t e = p + 1 < part_base[c + 1] ? rec[p + 1].start : cols[c].n;
    const Aux a = entry_of(r, pcoef, poly, p, e > r.start ? e - r.start : 0);
    aux[p] = a;
    zero_bound(a, words + word_base[c]);
  }
  for (uint64_t c = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; c < ncols; c += stride)
    for (uint64_t w = word_base[c] + (col_bits[c] >> 6); w < word_base[c + 1]; w++) words[w] = 0;
}

// k_pack over the columns of a batch: win_base[c] windows before column c's
template <typename T, bool POLY, bool SHORT>
__global__ void __launch_bounds__(kPackBlock, POLY ? 2 : kPackCtas)
    k_pack_multi(const EncCol* __restrict__ cols, const uint64_t* __restrict__ part_base,
                 const uint64_t* __restrict__ win_base, const uint64_t* __restrict__ word_base, uint32_t ncols,
                 uint64_t windows, uint32_t window, const Record* __restrict__ rec, const Aux* __restrict__ aux,
                 const PolyCoef* __restrict__ pcoef, const PolyAux* __restrict__ poly, uint64_t* __restrict__ words,
                 uint32_t lane_part) {
  __shared__ uint64_t zbuf[kPackWarps][kPackTile / 2];
  const uint32_t lane = threadIdx.x & 31u, wid = threadIdx.x >> 5;
  const uint64_t nw = (uint64_t)gridDim.x * kPackWarps;
  for (uint64_t k = (uint64_t)blockIdx.x * kPackWarps + wid; k < windows; k += nw) {
    const uint32_t c = find_col(win_base, ncols, k);
    const EncCol col = cols[c];
    const uint64_t pos = (k - win_base[c]) * window;
    const uint64_t p0 = part_base[c];
    pack_window<T, POLY, SHORT, true>(static_cast<const T*>(col.values), col.n, part_base[c + 1] - p0, pos, min(pos + window, col.n),
                         pos / col.L, rec + p0, aux + p0, POLY ? pcoef + p0 : nullptr, POLY ? poly + p0 : nullptr,
                         reinterpret_cast<uint32_t*>(words + word_base[c]), zbuf[wid], lane, lane_part);
  }
}

__global__ void k_part_col(const uint64_t* __restrict__ part_base, uint32_t ncols, uint64_t P,
                           uint32_t* __restrict__ part_col) {
  for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < P; p += (uint64_t)gridDim.x * blockDim.x)
    part_col[p] = find_col(part_base, ncols, p);
}

// exclusive prefix sum of the columns' stream words: each thread sums a contiguous run of columns,
// the CTA scans the run totals, then each thread writes its run's bases
constexpr int kWordBaseBlock = 1024;
__global__ void __launch_bounds__(kWordBaseBlock)
    k_word_bases(const uint64_t* __restrict__ col_bits, uint32_t ncols, uint64_t* __restrict__ word_base) {
  __shared__ uint64_t run[kWordBaseBlock];
  const uint32_t t = threadIdx.x;
  const uint64_t per = ((uint64_t)ncols + kWordBaseBlock - 1) / kWordBaseBlock;
  const uint32_t c0 = (uint32_t)min((uint64_t)t * per, (uint64_t)ncols);
  const uint32_t c1 = (uint32_t)min((uint64_t)c0 + per, (uint64_t)ncols);
  uint64_t s = 0;
  for (uint32_t c = c0; c < c1; c++) s += stream_words(col_bits[c]);
  run[t] = s;
  __syncthreads();
  for (uint32_t d = 1; d < kWordBaseBlock; d <<= 1) {
    const uint64_t add = t >= d ? run[t - d] : 0;
    __syncthreads();
    run[t] += add;
    __syncthreads();
  }
  uint64_t base = run[t] - s;
  for (uint32_t c = c0; c < c1; c++) {
    word_base[c] = base;
    base += stream_words(col_bits[c]);
  }
  if (t == kWordBaseBlock - 1) word_base[ncols] = run[t];
}

int grid_for(uint64_t items, int per_block, int max_blocks_per_sm) {
  const uint64_t need = (items + per_block - 1) / per_block;
  const uint64_t cap = (uint64_t)sm_count() * max_blocks_per_sm;
  return (int)(need < cap ? (need ? need : 1) : cap);
}

}  // namespace

int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) dev = 0;
  if (!cached[dev]) {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = v > 0 ? v : 1;
  }
  return cached[dev];
}

// the four polynomial phases over partitions [0, m) of the map, with their scratch (given: at least
// poly_fit_scratch_bytes(m) bytes the caller owns; nullptr: taken from the pool and released)
template <typename Map>
cudaError_t launch_poly_fit(const Map& map, int dtype, uint64_t m, Record* rec, uint64_t* lenbits, PolyCoef* pcoef,
                            uint32_t* max_b, cudaStream_t st, void* given = nullptr) {
  const uint64_t bm = (sizeof(PolyMom) * m + 255) & ~255ull, bp = (sizeof(PolyPlan) * m + 255) & ~255ull;
  char* scr = static_cast<char*>(given);
  cudaError_t e = given ? cudaSuccess : dev_alloc((void**)&scr, bm + bp + sizeof(PolyRange) * m, st);
  if (e != cudaSuccess) return e;
  PolyMom* mom = reinterpret_cast<PolyMom*>(scr);
  PolyPlan* plan = reinterpret_cast<PolyPlan*>(scr + bm);
  PolyRange* rng = reinterpret_cast<PolyRange*>(scr + bm + bp);
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_poly_ranges<Map>, kFitBlock, 0) != cudaSuccess || nb < 1)
    nb = 1;
  const uint64_t wb = (m + kFitWarps - 1) / kFitWarps;
  k_poly_moments<Map><<<grid_for(wb, 1, 8), kFitBlock, 0, st>>>(map, dtype, m, mom);
  k_poly_plan<Map><<<grid_for(m, 128, 8), 128, 0, st>>>(map, m, mom, plan);
  k_poly_ranges<Map><<<grid_for(wb, 1, nb), kFitBlock, 0, st>>>(map, dtype, m, plan, rng);
  k_poly_choose<Map><<<grid_for(m, 128, 8), 128, 0, st>>>(map, m, mom, plan, rng, rec, lenbits, pcoef, max_b);
  e = cudaGetLastError();
  if (!given) cudaFreeAsync(scr, st);
  return e;
}

// eight lanes per partition up to kFitTileVals values, sixteen up to 1023; a warp for partitions of any lengths
template <typename T>
void launch_fit_tiles(const T* values, uint64_t n, const uint64_t* starts, uint32_t L, uint64_t m, int ctas, int model,
                      Record* rec, uint64_t* lenbits, uint32_t* max_b, cudaStream_t st) {
  auto grid = [&](uint64_t per) { return grid_for((m + per - 1) / per, kFitWarps, ctas); };
  // short ones by fours while each of the warps has two groups of four at the least
  if (starts && n / m <= kFitShortMean && m >= 8ull * sm_count() * ctas * kFitWarps)
    k_fit_short<T><<<grid(4), kFitBlock, 0, st>>>(values, n, starts, m, model, rec, lenbits, max_b);
  else if (starts)
    k_fit<T, 32><<<grid(1), kFitBlock, 0, st>>>(values, n, starts, L, m, model, rec, lenbits, max_b);
  else if (L <= kFitTileVals)
    k_fit<T, 8><<<grid(4), kFitBlock, 0, st>>>(values, n, starts, L, m, model, rec, lenbits, max_b);
  else
    k_fit<T, 16><<<grid(2), kFitBlock, 0, st>>>(values, n, starts, L, m, model, rec, lenbits, max_b);
}

cudaError_t launch_fit(const void* values, int dtype, uint64_t n, const uint64_t* starts,
                       uint32_t L, uint64_t m, int model, Record* rec, uint64_t* lenbits, PolyCoef* pcoef,
                       uint32_t* max_b, cudaStream_t st) {
  if (model == LECO_MODEL_POLY && !pcoef) return cudaErrorInvalidValue;
  cudaError_t e = cudaMemsetAsync(max_b, 0, sizeof(uint32_t), st);
  if (e != cudaSuccess || m == 0) return e;
  if (model == LECO_MODEL_POLY) return launch_poly_fit(OneColumn{values, n, starts, L}, dtype, m, rec, lenbits, pcoef,
                                                        max_b, st);
  const uint32_t fc = encode_config_lookup(dtype).fit_ctas;
  const int ctas = fit_ctas_of(fc, kFitCtasPerSm);
  // partitions of at least 1024 values: two warps each (the second pass then stays in L2)
  if (!starts && L >= 1024) {
    k_fit_pairs<<<grid_for((m + kFitPairs - 1) / kFitPairs, 1, fit_ctas_of(fc, kPairCtas)), kFitBlock, 0, st>>>(
        values, dtype, n, starts, L, m, model, rec, lenbits, max_b);
    return cudaGetLastError();
  }
  if (dtype == LECO_U32)
    launch_fit_tiles(static_cast<const uint32_t*>(values), n, starts, L, m, ctas, model, rec, lenbits, max_b, st);
  else
    launch_fit_tiles(static_cast<const uint64_t*>(values), n, starts, L, m, ctas, model, rec, lenbits, max_b, st);
  return cudaGetLastError();
}

uint64_t offsets_scratch_elems(uint64_t m) {
  const uint64_t ntiles = (m + kPrefixTile - 1) / kPrefixTile;
  return m + ntiles + 1;  // exclusive offsets + tile prefixes + total
}

// exclusive scan of in[0..count) into out; *total (device) = the sum. scratch: ntiles+1 elems.
cudaError_t scan_u64(const uint64_t* in, uint64_t count, uint64_t* out, uint64_t* scratch,
                     uint64_t* total, cudaStream_t st) {
  if (count == 0) return cudaMemsetAsync(total, 0, sizeof(uint64_t), st);
  const uint64_t ntiles = (count + kPrefixTile - 1) / kPrefixTile;
  k_prefix_tiles<<<(unsigned)ntiles, kPrefixBlock, 0, st>>>(in, count, scratch);
  k_prefix_top<<<1, kPrefixBlock, 0, st>>>(scratch, ntiles, total);
  k_prefix_apply<<<(unsigned)ntiles, kPrefixBlock, 0, st>>>(in, count, scratch, out);
  return cudaGetLastError();
}

cudaError_t launch_offsets(Record* rec, const uint64_t* lenbits, uint64_t m, uint64_t* scratch,
                           uint64_t scratch_elems, uint64_t* total_out, cudaStream_t st) {
  (void)scratch_elems;
  if (m == 0) return cudaMemsetAsync(total_out, 0, sizeof(uint64_t), st);
  if (m <= kOneCtaParts) {
    k_offsets_one<<<1, kOneCtaBlock, 0, st>>>(rec, lenbits, (uint32_t)m, total_out);
    return cudaGetLastError();
  }
  uint64_t* off = scratch;
  uint64_t* tiles = scratch + m;
  cudaError_t e = scan_u64(lenbits, m, off, tiles, total_out, st);
  if (e != cudaSuccess) return e;
  k_set_offsets<<<grid_for(m, 256, 8), 256, 0, st>>>(rec, off, m);
  return cudaGetLastError();
}

cudaError_t launch_build_aux(const Record* rec, const PolyCoef* pcoef, uint64_t m, uint64_t n, Aux* aux,
                             PolyAux* poly, uint64_t total_bits, uint64_t* words, uint64_t nwords, uint32_t* status,
                             cudaStream_t st) {
  const uint64_t tail = total_bits >> 6, count = m + (words && nwords > tail ? nwords - tail : 0);
  if (count == 0) return status ? cudaMemsetAsync(status, 0, 4, st) : cudaSuccess;
  k_build_aux<<<grid_for(count, 256, 8), 256, 0, st>>>(rec, pcoef, m, n, aux, poly, total_bits, nwords, words, status);
  return cudaGetLastError();
}

template <typename T, bool POLY>
cudaError_t launch_pack_t(const void* values, uint64_t n, uint64_t m, uint32_t L, const TileDesc* tiles,
                          const Record* rec, const Aux* aux, const PolyCoef* pcoef, const PolyAux* poly,
                          uint32_t max_b, uint64_t* words, cudaStream_t st) {
  // 250M timestamps of ~570-value partitions packed in 650 us with windows of 1024 (which cut most partitions)
  // and 531 us with 4096; columns below 5M values come down to 256
  uint32_t window = pack_window(n, kPackWindow, kPackWindowMin, sm_count() * 128);
  // Fixed partitions: whole ones to a window, or a partition's windows from its start on, so that none is cut
  // where it need not be. Whole encodes, windows at any position -> this: 20M values in partitions of 1000 / 1500
  // / 2047 / 3000 159 / 180 / 160 / 151 -> 142 / 167 / 151 / 145 us, 150M of 1000 / 1500 563 / 760 -> 520 / 704.
  uint32_t period = window, per = 1;
  if (L && L <= window) {
    period = window -= window % L;
  } else if (L) {
    period = (uint32_t)min((uint64_t)L, n);
    per = (uint32_t)(((uint64_t)period + window - 1) / window);
  }
  const uint64_t nwin = (n + period - 1) / period * per;
  const uint32_t lane_part = POLY ? 0u : lane_part_of(n / m, window, max_b);
  const bool wide = max_b > 32;
  auto kern = lane_part ? (wide ? k_pack<T, POLY, !POLY, true> : k_pack<T, POLY, !POLY, POLY>)
                        : (wide ? k_pack<T, POLY, false, true> : k_pack<T, POLY, false, POLY>);
  kern<<<grid_for(nwin, kPackWarps, 8), kPackBlock, 0, st>>>(
      static_cast<const T*>(values), n, m, L, window, period, per, tiles, rec, aux, pcoef, poly,
      reinterpret_cast<uint32_t*>(words), lane_part);
  return cudaGetLastError();
}

cudaError_t launch_pack(const void* values, int dtype, uint32_t L, const TileDesc* tiles, const Record* rec,
                        const Aux* aux, const PolyCoef* pcoef, const PolyAux* poly, uint64_t m, uint64_t n,
                        uint32_t max_b, uint64_t* words, cudaStream_t st) {
  if (m == 0) return cudaSuccess;
  if (dtype == LECO_U32)
    return pcoef ? launch_pack_t<uint32_t, true>(values, n, m, L, tiles, rec, aux, pcoef, poly, max_b, words, st)
                 : launch_pack_t<uint32_t, false>(values, n, m, L, tiles, rec, aux, nullptr, nullptr, max_b, words, st);
  return pcoef ? launch_pack_t<uint64_t, true>(values, n, m, L, tiles, rec, aux, pcoef, poly, max_b, words, st)
               : launch_pack_t<uint64_t, false>(values, n, m, L, tiles, rec, aux, nullptr, nullptr, max_b, words, st);
}

cudaError_t launch_part_col(const uint64_t* part_base, uint32_t ncols, uint64_t P, uint32_t* part_col, cudaStream_t st) {
  if (P == 0) return cudaSuccess;
  k_part_col<<<grid_for(P, 256, 8), 256, 0, st>>>(part_base, ncols, P, part_col);
  return cudaGetLastError();
}

uint64_t poly_fit_scratch_bytes(uint64_t m) {
  return ((sizeof(PolyMom) * m + 255) & ~255ull) + ((sizeof(PolyPlan) * m + 255) & ~255ull) + sizeof(PolyRange) * m;
}

cudaError_t launch_fit_multi(const EncCol* cols, const uint64_t* part_base, const uint32_t* part_col, uint32_t ncols,
                             uint64_t P, int dtype, Record* rec, uint64_t* lenbits, PolyCoef* pcoef, uint32_t* max_b,
                             uint64_t values, uint32_t longest, uint32_t fit_ctas, cudaStream_t st,
                             void* poly_scratch) {
  cudaError_t e = cudaMemsetAsync(max_b, 0, sizeof(uint32_t) * (ncols ? ncols : 1), st);
  if (e != cudaSuccess || P == 0) return e;
  const int per_sm = fit_ctas_of(fit_ctas, kPairCtas);
  uint32_t parts = fit_parts(values, (uint64_t)sm_count() * per_sm * kFitPairs, longest, kFitTileVals);
  const bool mid = longest > kFitTileVals && longest <= kFitMidVals;
  if (mid && parts > 2) parts = 2;  // four at a time
  const int grid = grid_for((P + 7) / 8 * parts, kFitPairs, per_sm);
  auto launch = [&](auto value) {
    using T = decltype(value);
    auto kern = mid ? k_fit_multi<T, true, true> : parts > 1 ? k_fit_multi<T, true, false> : k_fit_multi<T, false, false>;
    kern<<<grid, kFitBlock, 0, st>>>(cols, part_base, part_col, P, parts, rec, lenbits, max_b);
  };
  if (dtype == LECO_U32)
    launch(uint32_t());
  else
    launch(uint64_t());
  e = cudaGetLastError();
  if (e == cudaSuccess && pcoef)
    e = launch_poly_fit(BatchColumns{cols, part_base, ncols}, dtype, P, rec, lenbits, pcoef, max_b, st, poly_scratch);
  return e;
}

uint64_t offsets_multi_scratch_elems(uint64_t P) { return P + (P + kPrefixTile - 1) / kPrefixTile + 2; }

cudaError_t launch_offsets_multi(Record* rec, const uint64_t* lenbits, const uint64_t* part_base,
                                 const uint32_t* part_col, uint32_t ncols, uint64_t P, uint64_t* scratch,
                                 uint64_t* col_bits, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(col_bits, 0, sizeof(uint64_t) * (ncols ? ncols : 1), st);
  if (e != cudaSuccess || P == 0) return e;
  uint64_t* off = scratch;
  uint64_t* tiles = scratch + P;
  uint64_t* total = scratch + offsets_multi_scratch_elems(P) - 1;
  e = scan_u64(lenbits, P, off, tiles, total, st);
  if (e != cudaSuccess) return e;
  k_set_offsets_multi<<<grid_for(P, 256, 8), 256, 0, st>>>(rec, off, lenbits, part_base, part_col, P, col_bits);
  return cudaGetLastError();
}

cudaError_t launch_aux_multi(const Record* rec, const PolyCoef* pcoef, const EncCol* cols, const uint64_t* part_base,
                             const uint32_t* part_col, const uint64_t* word_base, const uint64_t* col_bits,
                             uint32_t ncols, uint64_t P, Aux* aux, PolyAux* poly, uint64_t* words, cudaStream_t st) {
  if (P == 0 && ncols == 0) return cudaSuccess;
  k_aux_multi<<<grid_for(P > ncols ? P : ncols, 256, 8), 256, 0, st>>>(rec, pcoef, cols, part_base, part_col, word_base,
                                                                       col_bits, ncols, P, aux, poly, words);
  return cudaGetLastError();
}

cudaError_t launch_word_bases(const uint64_t* col_bits, uint32_t ncols, uint64_t* word_base, cudaStream_t st) {
  k_word_bases<<<1, kWordBaseBlock, 0, st>>>(col_bits, ncols, word_base);
  return cudaGetLastError();
}

template <typename T, bool POLY>
cudaError_t launch_pack_multi_t(const EncCol* cols, const uint64_t* part_base, const uint64_t* win_base,
                                const uint64_t* word_base, uint32_t ncols, uint64_t windows, uint32_t window, uint32_t lane_part,
                                const Record* rec, const Aux* aux, const PolyCoef* pcoef, const PolyAux* poly,
                                uint64_t* words, cudaStream_t st) {
  auto kern = lane_part ? k_pack_multi<T, POLY, !POLY> : k_pack_multi<T, POLY, false>;
  kern<<<grid_for(windows, kPackWarps, 8), kPackBlock, 0, st>>>(
      cols, part_base, win_base, word_base, ncols, windows, window, rec, aux, pcoef, poly, words, lane_part);
  return cudaGetLastError();
}

cudaError_t launch_pack_multi(const EncCol* cols, const uint64_t* part_base, const uint64_t* win_base,
                              const uint64_t* word_base, uint32_t ncols, uint64_t windows, int dtype, uint32_t window, uint64_t mean,
                              const Record* rec, const Aux* aux, const PolyCoef* pcoef, const PolyAux* poly,
                              uint64_t* words, cudaStream_t st) {
  if (windows == 0) return cudaSuccess;
  const uint32_t lp = pcoef ? 0u : lane_part_of(mean, window, 0);
  if (dtype == LECO_U32)
    return pcoef ? launch_pack_multi_t<uint32_t, true>(cols, part_base, win_base, word_base, ncols, windows, window, lp, rec,
                                                       aux, pcoef, poly, words, st)
                 : launch_pack_multi_t<uint32_t, false>(cols, part_base, win_base, word_base, ncols, windows, window, lp,
                                                        rec, aux, nullptr, nullptr, words, st);
  return pcoef ? launch_pack_multi_t<uint64_t, true>(cols, part_base, win_base, word_base, ncols, windows, window, lp, rec,
                                                     aux, pcoef, poly, words, st)
               : launch_pack_multi_t<uint64_t, false>(cols, part_base, win_base, word_base, ncols, windows, window, lp, rec,
                                                      aux, nullptr, nullptr, words, st);
}

}  // namespace leco
