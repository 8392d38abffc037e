// Batched point lookups (§3.3 Decoder): one thread per requested position.
//
// Value at position i of partition p: pred_p(i - start_p) + unzigzag(bits [off_p + b_p (i -
// start_p), +b_p)) mod 2^64. The prediction comes from the decode table (integer grid) and falls
// back to binary64 for records whose exact flag did not verify.
#include "leco_internal.cuh"

namespace leco {

namespace {

constexpr int kBlock = 256;

// Scattered loads are what a lookup costs: the L1 takes about one 32-byte sector per clock and SM, and a column
// that fits L2 is bound by that. So a lookup takes each thing it needs in one load: the first partition
// and the partition count of its tile, four starts at a time, the whole decode-table entry, and the second
// residual word only where the field crosses into it: 5M lookups in 100M 32-bit timestamps (variable
// partitions) 129 -> 98 us against a binary search, two 16-byte entry loads and both words always.

struct Load32 {
  uint64_t x[4];
};
__device__ __forceinline__ Load32 load32(const void* p) {  // 32-byte aligned
  Load32 r;
  asm("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];" : "=l"(r.x[0]), "=l"(r.x[1]), "=l"(r.x[2]), "=l"(r.x[3]) : "l"(p));
  return r;
}

// Variable partitions: the largest p with starts[p] <= i among the partitions touching i's scan tile
// (its descriptor names the first and how many), searched by groups of four starts: the first group is
// guessed from i's place in the tile, the second is a neighbour, then the middle.
struct PartSearch {
  uint64_t p0;
  uint32_t lo, hi, guess;  // relative to p0: starts[lo] <= i, starts[hi] > i
  __device__ __forceinline__ void begin(const ColumnView& c, uint64_t i) {
    const uint4 d = __ldg(reinterpret_cast<const uint4*>(c.tiles + i / kScanTile));
    p0 = (uint64_t)d.y << 32 | d.x;
    lo = 0;
    hi = d.z;
    guess = ((uint32_t)(i % kScanTile) * hi) / (uint32_t)kScanTile;  // a tile touches at most kScanTile partitions
  }
  __device__ __forceinline__ bool open() const { return hi - lo > 1; }
  __device__ __forceinline__ const uint64_t* group(const ColumnView& c) const { return c.starts + ((p0 + guess) & ~3ull); }
  __device__ __forceinline__ void take(const Load32& s, uint64_t i, uint32_t step) {
    const int32_t first = (int32_t)((uint32_t)((p0 + guess) & ~3ull) - (uint32_t)p0);  // may precede p0
    const uint32_t was = lo;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int32_t at = first + j;
      if (at > (int32_t)lo && at < (int32_t)hi) {
        if (s.x[j] <= i)
          lo = (uint32_t)at;
        else
          hi = (uint32_t)at;
      }
    }
    guess = step ? (lo + hi) >> 1 : lo != was ? lo + 1 : hi - 1;
  }
};

// fixed partitions: the one holding position i (< n)
__device__ __forceinline__ uint64_t fixed_part(const ColumnView& c, uint64_t i) {
  return c.n <= 0xFFFFFFFFull ? (uint32_t)i / c.L : i / c.L;
}

// partition holding position i (< n)
__device__ __forceinline__ uint64_t find_part(const ColumnView& c, uint64_t i) {
  if (!c.starts) return fixed_part(c, i);
  PartSearch s;
  s.begin(c, i);
  for (uint32_t step = 0; s.open(); step++) s.take(load32(s.group(c)), i, step);
  return s.p0 + s.lo;
}

__device__ __forceinline__ Aux load_aux(const Aux* __restrict__ aux, uint64_t p) {
  const Load32 v = load32(aux + p);
  Aux a;
  a.A = (int64_t)v.x[0];
  a.B = (int64_t)v.x[1];
  a.start = v.x[2];
  a.word3 = v.x[3];
  return a;
}

// U independent lookups per thread and iteration: their loads (index, decode-table entry, residual words) are
// issued together, so each thread keeps several memory round trips in flight. VAR (variable partitions) is a kernel
// of its own, two lookups per thread in 64 registers (four CTAs per SM) where a fixed column takes four in 76 (three):
// with the search behind a branch of one kernel both held 118 registers, two CTAs per SM, and fixed columns paid for
// a search they never run. 10M lookups in 200M values of fixed partitions 213 -> 193 us, 5M in 20M values 76 -> 63 us;
// variable partitions: 5M in 1M near-linear values 35 -> 29 us, 5M in 100M timestamps 98 -> 82 us, 10M in 100M piecewise
// values 244 -> 176 us (three or four lookups per thread: 94 / 96 us on the timestamps, 215 / 242 us on the piecewise).
constexpr int kUnroll = 4, kVarUnroll = 2;

template <typename T, bool VAR>
__global__ void __launch_bounds__(kBlock)
    k_random_access(const ColumnView c, const uint64_t* __restrict__ idx, uint64_t k,
                    T* __restrict__ out) {
  constexpr int U = VAR ? kVarUnroll : kUnroll;
  const uint64_t stride = (uint64_t)gridDim.x * kBlock;
  for (uint64_t base = (uint64_t)blockIdx.x * kBlock + threadIdx.x; base < k; base += stride * U) {
    uint64_t i[U], p[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint64_t q = base + (uint64_t)u * stride;
      i[u] = q < k ? __ldg(idx + q) : 0;
      ok[u] = q < k && i[u] < c.n;
    }
    if (VAR) {  // the searches of the thread's lookups step together
      PartSearch f[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        f[u].begin(c, ok[u] ? i[u] : 0);
        if (!ok[u]) f[u].hi = 0;
      }
      bool more = true;
      for (uint32_t step = 0; more; step++) {
        more = false;
        Load32 s[U];
#pragma unroll
        for (int u = 0; u < U; u++)
          if (f[u].hi > f[u].lo + 1) s[u] = load32(f[u].group(c));
#pragma unroll
        for (int u = 0; u < U; u++) {
          if (f[u].hi <= f[u].lo + 1) continue;
          f[u].take(s[u], i[u], step);
          more = more || f[u].open();
        }
      }
#pragma unroll
      for (int u = 0; u < U; u++) p[u] = ok[u] ? f[u].p0 + f[u].lo : 0;
    } else {
#pragma unroll
      for (int u = 0; u < U; u++) p[u] = ok[u] ? fixed_part(c, i[u]) : 0;
    }
    Aux a[U];
#pragma unroll
    for (int u = 0; u < U; u++) a[u] = load_aux(c.aux, ok[u] ? p[u] : 0);
    uint64_t z[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint64_t x = i[u] - a[u].start;
      const uint32_t b = w3_b(a[u].word3);
      z[u] = ok[u] ? read_field(c.words, w3_off(a[u].word3) + x * b, b) : 0;
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
      const uint64_t q = base + (uint64_t)u * stride;
      if (q >= k) continue;
      if (!ok[u]) {
        out[q] = 0;
        atomicOr(c.status, kStatIndexRange);
        continue;
      }
      const int64_t pred = predict_aux(a[u], c.rec, c.poly, p[u], i[u] - a[u].start);
      out[q] = (T)((uint64_t)pred + (uint64_t)zz_decode(z[u]));
    }
  }
}

// Lookups of several columns in one launch (a serving batch): index q reads column col[q]; results
// are widened to 64 bits (a 32-bit column's value is zero-extended).
__global__ void __launch_bounds__(kBlock)
    k_lookup_multi(const ColumnView* __restrict__ views, const uint32_t* __restrict__ col,
                   const uint64_t* __restrict__ idx, uint64_t k, uint64_t* __restrict__ out) {
  for (uint64_t q = (uint64_t)blockIdx.x * kBlock + threadIdx.x; q < k; q += (uint64_t)gridDim.x * kBlock) {
    const ColumnView c = views[col[q]];
    const uint64_t i = __ldg(idx + q);
    if (i >= c.n) {
      out[q] = 0;
      atomicOr(c.status, kStatIndexRange);
      continue;
    }
    const uint64_t p = find_part(c, i);
    const Aux a = load_aux(c.aux, p);
    const uint64_t x = i - a.start;
    const uint32_t b = w3_b(a.word3);
    const uint64_t z = read_field(c.words, w3_off(a.word3) + x * b, b);
    const uint64_t v = (uint64_t)predict_aux(a, c.rec, c.poly, p, x) + (uint64_t)zz_decode(z);
    out[q] = c.dtype == LECO_U32 ? (v & 0xFFFFFFFFull) : v;
  }
}

int grid_for(uint64_t items, int per_block, int max_blocks_per_sm) {
  const uint64_t need = (items + per_block - 1) / per_block;
  const uint64_t cap = (uint64_t)sm_count() * max_blocks_per_sm;
  return (int)(need < cap ? (need ? need : 1) : cap);
}

}  // namespace

cudaError_t launch_random_access(const ColumnView& c, const uint64_t* idx, uint64_t k, void* out,
                                 cudaStream_t st) {
  if (k == 0) return cudaSuccess;
  const int u = c.starts ? kVarUnroll : kUnroll, grid = grid_for((k + u - 1) / u, kBlock, 8);
  if (c.dtype == LECO_U32)
    (c.starts ? k_random_access<uint32_t, true> : k_random_access<uint32_t, false>)<<<grid, kBlock, 0, st>>>(
        c, idx, k, (uint32_t*)out);
  else
    (c.starts ? k_random_access<uint64_t, true> : k_random_access<uint64_t, false>)<<<grid, kBlock, 0, st>>>(
        c, idx, k, (uint64_t*)out);
  return cudaGetLastError();
}

cudaError_t launch_lookup_multi(const ColumnView* views, const uint32_t* col, const uint64_t* idx, uint64_t k,
                                uint64_t* out, cudaStream_t st) {
  if (k == 0) return cudaSuccess;
  k_lookup_multi<<<grid_for(k, kBlock, 8), kBlock, 0, st>>>(views, col, idx, k, out);
  return cudaGetLastError();
}

}  // namespace leco
