// Host-side choices of launch shapes (no CUDA calls here).
#pragma once

#include <stdint.h>

#include <atomic>

namespace leco {

// CTAs per SM of one kernel by device and shared-memory size: asked once for each, because the driver calls
// that answer cost more than a launch. A program's columns differ in width and so in stage size, and their
// scans alternate: with room for one size per device every scan asked again (three columns of
// 1M values in turn took 27.6 us a query, columns of one width 25.8; now both the same). A slot per KiB of shared memory
// (widths differ by at least that, two stages of 512 bytes); a size that shares a slot is asked again when
// the other was there last. Any number of threads.
class ResidentCache {
 public:
  // ask(): a positive count, or anything else for "not known" (returned, and not kept)
  template <typename F>
  int get(int dev, uint32_t smem, F ask) {
    std::atomic<uint32_t>* slot =
        dev >= 0 && dev < kDevices && smem < (1u << 24) ? &slots_[dev][(smem >> 10) % kSizes] : nullptr;
    const uint32_t seen = slot ? slot->load(std::memory_order_relaxed) : 0u;
    if ((seen & 0xFFu) && (seen >> 8) == smem) return (int)(seen & 0xFFu);
    const int n = ask();
    if (slot && n > 0 && n < 256) slot->store(smem << 8 | (uint32_t)n, std::memory_order_relaxed);
    return n;
  }

 private:
  static constexpr int kDevices = 64, kSizes = 256;
  std::atomic<uint32_t> slots_[kDevices][kSizes] = {};
};

constexpr uint32_t kPackWindowMin = 256;

// Positions per warp of the packer: the most (window), halved down to `least` until there are `wanted` windows, so
// that a few thousand values do not wait for one warp and the last wave weighs little. A column wants four windows
// per resident warp (32 per SM), a batch one, since each of its windows searches its column: four columns of 3000
// values in partitions of 64, windows of 4096 -> 256 positions: 52 -> 7 us; 20 columns of 8M values in partitions of
// 256 36 -> 28 us; 16M 32-bit values 38 -> 34 us (four per warp: 46 us).
inline uint32_t pack_window(uint64_t values, uint32_t window, uint32_t least, int wanted) {
  while (window > least && values / window < (uint64_t)wanted) window /= 2;
  return window;
}

constexpr uint32_t kLaneBits = 2048;  // most bits of a partition that one lane packs

// Values up to which the packer gives a whole partition to one lane (k_pack's SHORT kernel), by the column's mean,
// the window and the widest partition (max_b; 0: not known); 0: the kernel that has no such lanes, a warp on one
// partition after another. Above a mean of 96 only the shortest ones gain, above 224 there are too few of them for the
// registers they cost; a small window holds few partitions, so that a lane's longer chain is not hidden. Packer of
// 2.7M partitions of 1 .. 15 values 1335 -> 178 us, 400K of 1 .. 99 268 -> 185 us, 110K of which nine in ten have
// 1 .. 19 and the others 500 .. 2999 values 229 -> 107 us, 5M of 4 2774 -> 151 us; 133K of 1 .. 299 values lose by
// it, 122 -> 131 us.
inline uint32_t lane_part_of(uint64_t mean, uint32_t window, uint32_t max_b) {
  const uint32_t most = mean * max_b > kLaneBits + kLaneBits / 2 ? 0u : mean <= 96 ? 128u : mean <= 224 ? 32u : 0u;
  return most < window / 8 ? most : window / 8;
}

// Parts that a group of eight partitions of a batched fit is dealt out in, so that the longest item is at most
// half of what a pair of warps has to fit (values / pairs). longest: the longest partition; those up to `tile`
// values are fitted eight at a time and stay together.
inline uint32_t fit_parts(uint64_t values, uint64_t pairs, uint32_t longest, uint32_t tile) {
  uint32_t parts = 1;
  if (longest > tile)
    while (parts < 8 && (uint64_t)(8 / parts) * longest * 2 * pairs > values) parts *= 2;
  return parts;
}

// CTAs per SM of a fit, at most `most` (what its registers allow): 2 where the tuning table asks for it (fewer keep
// more of each partition in L2 for the second pass), else as many as there can be. The batched fit holds three, so that
// 3 and 4 are the same to it, and the tuner tries only what differs.
constexpr uint32_t kFitCtasTried[] = {2, 3};
inline int fit_ctas_of(uint32_t asked, int most) { return asked == 2 && most > 2 ? 2 : most; }

}  // namespace leco
