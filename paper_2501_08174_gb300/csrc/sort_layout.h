// Sizes of the radix sorts of the binning: the items of a tile, the digits of a key and the
// scratch of a sort.
// Plain C++, so that a program on the CPU can check them.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>

namespace ocgs {
namespace sort_layout {

// 384 threads x 18 items at three blocks per SM (56 registers, 69 KB) was the fastest of
// 256 to 512 threads x 10 to 24 items: 36 resident warps hide the ranking's shared-memory
// latency and few tiles keep the look-back short (tile sorts of 500k surfels x 16 views,
// 28 M pairs: 376 us against 400 to 516 with the others, 584 with a histogram, a scan and
// a scatter kernel per digit; depth sort of 8 M records: 230 against 390).
constexpr int kRadixThreads = 384;
constexpr int kRadixItems = 18;
// Where tiles of 18 items would leave SMs idle, tiles of 4: a pass over few items is the
// latency of one tile, and that of its serial ranking rounds (a pass over 2,000 records: 8.2
// -> 5.5 us; the depth sort of 100k: 52 -> 43 us).
constexpr int kSmallItems = 4;
constexpr uint32_t kSmallSort = 152u * kRadixThreads * kSmallItems;  // at most one small tile per SM

// Tiles of a sort of n items.  Not monotonic: there are fewer just above kSmallSort than at it.
inline size_t tile_count(uint32_t n) {
  const size_t tile = (size_t)kRadixThreads * (n <= kSmallSort ? kSmallItems : kRadixItems);
  return ((size_t)n + tile - 1) / tile;
}
// The most tiles a sort of any m <= n items has.
inline size_t tile_bound(uint32_t n) { return std::max(tile_count(n), tile_count(std::min(n, kSmallSort))); }

// Digits of a sort of n_bits key bits: equal widths of 4 to 8 bits.  (Two digits of 10
// bits instead of three of 7 took 17.6 against 6.0 ms on 480k tiles: runs of a few items
// per digit and tile, and four times the look-back words.)
constexpr int kMinDigit = 4, kMaxDigit = 8;
struct DigitPlan {
  int passes, bits;
};
constexpr DigitPlan digit_plan(int n_bits) {
  const int passes = (n_bits + kMaxDigit - 1) / kMaxDigit;
  return DigitPlan{passes, std::max(kMinDigit, (n_bits + passes - 1) / passes)};
}

// Scratch words of a sort: the digit positions of every pass, 64 words of counters, and one
// look-back word per pass, tile and digit.
constexpr size_t kCounterWords = 64;
inline size_t scratch_words(size_t tiles, int passes, int bits) {
  const size_t R = (size_t)1 << bits;
  return (size_t)passes * R + kCounterWords + (size_t)passes * tiles * R;
}
// Bytes a sort of n items uses.
inline size_t bytes_used(uint32_t n, int passes, int bits) {
  return sizeof(uint32_t) * scratch_words(tile_count(n), passes, bits);
}
// Bytes that hold the scratch of a sort of any m <= n items.
inline size_t bytes_for(uint32_t n, int passes, int bits) {
  return sizeof(uint32_t) * scratch_words(tile_bound(n), passes, bits);
}

}  // namespace sort_layout
}  // namespace ocgs
