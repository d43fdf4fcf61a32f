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

// Dynamic shared memory for the CTAs (of at most 64 registers a thread) of a kernel that is
// bound per SM and that programmatic launch may place while the kernel before it
// drains: `bytes`, or so much more that an SM holds no more of them than their even
// share.  Otherwise the SMs that drain first take far more than the others (a
// convolution of 50 and 300000 values over 5 levels: 1918 us, 1239 by plain launches,
// whose empty levels cost 75 us in a call of one level).  More CTAs than fit at once
// are placed as they end.
constexpr int SM_SMEM = 228 * 1024, CTA_SMEM_MAX = 226 * 1024;  // (1 KB for static arrays)
inline int even_share_smem(int bytes, int ctas, int threads, int sms) {
  const int share = (ctas + sms - 1) / sms, fit = std::min(1024 / threads, 32);
  if (share >= fit) return bytes;
  return std::max(bytes, std::min(CTA_SMEM_MAX, (SM_SMEM / share - 1024) & ~1023));
}

// The affine fit's stream over B's rows (k_fit_stream): a thread per sample, the
// samples' values of A for STREAM_K indices at a time, a ring of whole rows of B.
constexpr int STREAM_THREADS = 1024;
constexpr int STREAM_K = 16;
constexpr int STREAM_LD = STREAM_THREADS + 1;
constexpr int STREAM_A_FLOATS = (STREAM_K * STREAM_LD + 31) & ~31;
constexpr int STREAM_MAX_STAGES = 4;
constexpr int STREAM_SMEM = 220 * 1024;

// Ranges of the contraction for the stream (0: k_fit_samples) and the stages of its
// ring, where B's rows are 16-byte aligned and N a multiple of 4.  It needs a thread
// per sample and room for the partial sums (part_floats), and reads all of B where
// k_fit_samples reads a sector per term: B's rows at the copy rate cost less up to
// about 26 columns per sample (1024 samples, in us, stream with merge against a
// block per sample: n = 16384 246 / 285, 8192 91 / 136, 4096 63 / 70); below 4 M terms
// the merge costs more than the scattered reads.
inline int fit_stream_ranges(int64_t N, int64_t K, int64_t n_fit, int n_p, int64_t part_floats,
                             int sms, int* stages) {
  if (n_fit > STREAM_THREADS || n_fit * K < (4 << 20) || N > 16 * n_fit) return 0;
  const int64_t n = (STREAM_SMEM / 4 - STREAM_A_FLOATS) / N;
  if (n < 2) return 0;
  *stages = static_cast<int>(std::min<int64_t>(n, STREAM_MAX_STAGES));
  const int64_t room = part_floats / ((n_p + 1) * n_fit);
  const int64_t ranges = std::min<int64_t>(std::min<int64_t>(sms, K / STREAM_K), room);
  return ranges < 16 ? 0 : static_cast<int>(ranges);
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
