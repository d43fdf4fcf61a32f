// Host arithmetic of the launches, free of CUDA.
#pragma once
#include <algorithm>
#include <atomic>
#include <cstdint>

namespace pn {

// Tiles of the busiest of n CTAs that share out x.
inline int64_t tiles_owned(int64_t x, int64_t n) { return (x + n - 1) / n; }

// CTAs of `ctas` >= 2 that take operand A in a launch that builds xa >= 1 tiles of A
// and xb >= 1 of B, each CTA of one operand only: the split whose busiest CTA owns
// fewest tiles.  A's share grows as n falls and B's as it rises, and at the
// proportional share both are the average, so the best whole number is next to it.
inline int image_split(int64_t xa, int64_t xb, int ctas) {
  const int64_t below = static_cast<int64_t>(ctas) * xa / (xa + xb);
  const auto worst = [&](int64_t n) {
    return std::max(tiles_owned(xa, n), tiles_owned(xb, ctas - n));
  };
  const int64_t lo = std::min<int64_t>(std::max<int64_t>(below, 1), ctas - 1);
  const int64_t hi = std::min<int64_t>(below + 1, ctas - 1);
  return static_cast<int>(worst(hi) < worst(lo) ? hi : lo);
}

// The devices (0 .. 63) for which something has been done once; safe between threads.
class DeviceSet {
 public:
  bool has(int dev) const { return known(dev) && (bits_.load(std::memory_order_acquire) >> dev) & 1u; }
  void add(int dev) {
    if (known(dev)) bits_.fetch_or(uint64_t(1) << dev, std::memory_order_release);
  }

 private:
  static bool known(int dev) { return dev >= 0 && dev < 64; }
  std::atomic<uint64_t> bits_{0};
};

}  // namespace pn
