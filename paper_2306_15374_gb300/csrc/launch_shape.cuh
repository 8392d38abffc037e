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

}  // namespace leco
