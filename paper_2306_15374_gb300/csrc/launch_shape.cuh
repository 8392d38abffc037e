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

// Parts that a group of eight partitions of a batched fit is dealt out in, so that the longest item is at most
// half of what a pair of warps has to fit (values / pairs). longest: the longest partition; those up to `tile`
// values are fitted eight at a time and stay together.
inline uint32_t fit_parts(uint64_t values, uint64_t pairs, uint32_t longest, uint32_t tile) {
  uint32_t parts = 1;
  if (longest > tile)
    while (parts < 8 && (uint64_t)(8 / parts) * longest * 2 * pairs > values) parts *= 2;
  return parts;
}

}  // namespace leco
