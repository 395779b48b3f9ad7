// Decoupled look-back of the single-pass sorts and scans (Merrill and Garland,
// "Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016): a block
// publishes its tile's count, adds up the words of the tiles before it until one
// holds a running total, and publishes its own.  Tiles are handed out by a counter,
// so the tiles a block waits for are resident and never wait for a later one.  A
// wait that reaches kSpinLimit polls all the same is given up; the caller then
// counts the earlier items itself, so no result depends on a wait.
#pragma once

#include "common.cuh"

namespace ocgs {
namespace lookback {

constexpr unsigned kFull = 0xffffffffu;
// (A build with 0 gives up every look-back at once, so that the counting is what runs.)
#ifndef OCGS_SPIN_LIMIT
#define OCGS_SPIN_LIMIT (1u << 20)
#endif
constexpr uint32_t kSpinLimit = OCGS_SPIN_LIMIT;
constexpr int kLookBack = 16;  // tiles per round trip of a look-back (4 to 32 measured within 3 %)

template <typename T>
__device__ __forceinline__ T warp_inclusive_scan(T v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T t = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Word of one tile (and digit): 0 = nothing yet, count_word(c) = the tile's count c (at most
// kMaxTileCount), total_word(t) = the total t of the tiles up to and with it.
constexpr int kMaxTileCount = 8192;
__device__ __forceinline__ uint32_t count_word(uint32_t c) { return 1u + c; }
__device__ __forceinline__ uint32_t total_word(uint32_t t) { return (uint32_t)(kMaxTileCount + 2) + t; }

__device__ __forceinline__ uint32_t load_word(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void store_word(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Sum of the tiles before `tile` for this thread's digit (words: the digit's column,
// R apart).  False if the wait was given up.
template <int R>
__device__ __forceinline__ bool look_back(const uint32_t* words, uint32_t tile, uint32_t* excl) {
  if (kSpinLimit == 0u && tile > 0u) return false;
  uint32_t sum = 0, polls = 0;
  int64_t t = (int64_t)tile - 1;
  while (t >= 0) {
    uint32_t w[kLookBack];
#pragma unroll
    for (int k = 0; k < kLookBack; ++k) w[k] = t - k >= 0 ? load_word(words + (t - k) * R) : 0u;
    int used = 0;
#pragma unroll
    for (int k = 0; k < kLookBack; ++k) {
      if (used != k || w[k] == 0u) continue;
      if (w[k] > (uint32_t)kMaxTileCount + 1u) {
        *excl = sum + (w[k] - total_word(0u));
        return true;
      }
      sum += w[k] - 1u;
      used = k + 1;
    }
    t -= used;
    if (used == 0 && ++polls > kSpinLimit) return false;
  }
  *excl = sum;
  return true;
}

// The same for one word per tile, by a whole warp (every lane calls it and gets the result):
// 128 tiles per round trip.
__device__ __forceinline__ bool look_back_warp(const uint32_t* words, uint32_t tile, int lane, uint32_t* excl) {
  if (kSpinLimit == 0u && tile > 0u) return false;
  uint32_t sum = 0, polls = 0;
  int64_t t = (int64_t)tile - 1;
  while (t >= 0) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = t - (k * 32 + lane);
      w[k] = i >= 0 ? load_word(words + i) : total_word(0u);  // before the first tile: a total of 0
    }
    int used = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (used != 32 * k) break;  // (uniform)
      const unsigned none = __ballot_sync(kFull, w[k] == 0u);
      const unsigned tot = __ballot_sync(kFull, w[k] > (uint32_t)kMaxTileCount + 1u);
      const int first_none = none ? __ffs(none) - 1 : 32, first_tot = tot ? __ffs(tot) - 1 : 32;
      const int take = min(first_none, first_tot);
      uint32_t c = lane < take ? w[k] - 1u : 0u;
      if (lane == first_tot && first_tot < first_none) c = w[k] - total_word(0u);
      sum += __reduce_add_sync(kFull, c);
      if (first_tot < first_none) {
        *excl = sum;
        return true;
      }
      used += take;
    }
    t -= used;
    if (used == 0 && ++polls > kSpinLimit) return false;
  }
  *excl = sum;
  return true;
}

}  // namespace lookback
}  // namespace ocgs
