// Tile binning: the stable LSD radix sort of 32-bit keys, duplication of each
// visible (view, Gaussian) record into its tiles and the per-tile [start, end)
// ranges.
//
// Order of the (tile, Gaussian) list (the front-to-back order of Sec. 4.3):
// records are first sorted by centre depth (stable, so equal depths keep the
// ascending (view, Gaussian) index), duplicated in that order, and then
// stably sorted by global tile id.  Within a tile the list is therefore in
// ascending (depth, Gaussian index) order, and only ceil(log2 tiles) key bits
// are sorted per pair instead of tile+depth bits.
#include "lookback.cuh"
#include "sort_layout.h"

#include <algorithm>
#include <type_traits>

namespace ocgs {
namespace {
using namespace lookback;
using namespace sort_layout;

// ------------------------------------------------------------------ radix sort
// Stable LSD sort, one kernel per digit (the single-pass scatter with decoupled
// look-back of Adinets and Merrill, "Onesweep", 2022; see lookback.cuh): a first
// kernel reads the keys once and counts the digits of every pass; each pass then
// reads its items once and writes them once, a block ordering its tile by digit in
// shared memory.  A look-back that is given up is replaced by counting the digits
// of all earlier keys.
//
// What bounds it: HBM at full size (16 bytes per item and pass), the launch and
// the look-back latency below about a million items.
// (The sizes of a tile: sort_layout.h.)
constexpr int kRadixBlocks = 3;  // resident per SM
constexpr int kRadixWarps = kRadixThreads / 32;
static_assert(kRadixThreads * kRadixItems <= kMaxTileCount, "look-back words");

// Where the keys of a sort come from: an array, or (queue orders) the tiles' pair counts.
struct ArrayKeys {
  const uint32_t* keys;
  __device__ __forceinline__ uint32_t operator()(uint32_t i) const { return keys[i]; }
};
struct QueueKeys {
  const uint2* ranges;
  const uint2* ranges2;  // optional second segment of each tile's list
  __device__ __forceinline__ uint32_t operator()(uint32_t i) const {
    const uint2 r = ranges[i];
    uint32_t len = r.y - r.x;
    if (ranges2) {
      const uint2 q = ranges2[i];
      len += q.y - q.x;
    }
    return queue_class(len);
  }
};

// Exclusive scan of PER values per thread over a block of kRadixThreads; returns
// this thread's first prefix.  s_w: one word per warp, free to reuse after a barrier.
template <int PER>
__device__ __forceinline__ uint32_t block_exclusive(const uint32_t (&v)[PER], uint32_t* s_w) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t sum = 0;
#pragma unroll
  for (int k = 0; k < PER; ++k) sum += v[k];
  const uint32_t inc = warp_inclusive_scan<uint32_t>(sum, lane);
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  uint32_t carry = 0;
#pragma unroll
  for (int w = 0; w < kRadixWarps; ++w) carry += w < warp ? s_w[w] : 0u;
  return carry + inc - sum;
}

// Counts the digits of every pass (hist [PASSES][1 << BITS], zeroed); the last
// block to finish turns each pass's counts into first positions.  DROP: keys
// 0xffffffff are left out of the sort, and *n_valid gets the number of the others.
template <class Keys, int BITS, int PASSES, bool DROP>
__global__ void __launch_bounds__(kRadixThreads) radix_hist_kernel(const Keys keys, uint32_t n,
                                                                   const uint32_t* __restrict__ d_n, uint32_t* hist,
                                                                   uint32_t* done, uint32_t* n_valid) {
  constexpr int R = 1 << BITS, PER = (R + kRadixThreads - 1) / kRadixThreads;
  __shared__ uint32_t h[PASSES * R];
  __shared__ uint32_t s_w[kRadixWarps];
  __shared__ bool s_last;
  if (d_n) n = min(n, *d_n);  // device-side count (capacity launches)
  for (int i = threadIdx.x; i < PASSES * R; i += kRadixThreads) h[i] = 0;
  __syncthreads();
  auto count = [&](uint32_t k) {
    if (DROP && k == 0xffffffffu) return;
#pragma unroll
    for (int p = 0; p < PASSES; ++p) atomicAdd(&h[p * R + ((k >> (p * BITS)) & (R - 1))], 1u);
  };
  const uint32_t stride = gridDim.x * kRadixThreads, first = blockIdx.x * kRadixThreads + threadIdx.x;
  if constexpr (std::is_same<Keys, ArrayKeys>::value) {  // arena buffers: 16-byte aligned
    for (uint64_t i = first; 4 * i + 3 < n; i += stride) {
      const uint4 k = reinterpret_cast<const uint4*>(keys.keys)[i];
      count(k.x);
      count(k.y);
      count(k.z);
      count(k.w);
    }
    if (first < (n & 3u)) count(keys((n & ~3u) + first));
  } else {
    for (uint64_t i = first; i < n; i += stride) count(keys((uint32_t)i));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < PASSES * R; i += kRadixThreads)
    if (h[i]) atomicAdd(&hist[i], h[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
#pragma unroll
  for (int p = 0; p < PASSES; ++p) {
    uint32_t c[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int d = threadIdx.x * PER + k;
      c[k] = d < R ? __ldcg(hist + p * R + d) : 0u;
    }
    uint32_t e = block_exclusive<PER>(c, s_w);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int d = threadIdx.x * PER + k;
      if (d < R) hist[p * R + d] = e;
      e += c[k];
    }
    if (DROP && p == 0 && threadIdx.x == kRadixThreads - 1) *n_valid = e;
    __syncthreads();
  }
}

// One pass.  Warp w of a block owns the contiguous slice [w * 32 * kRadixItems, ...)
// of its tile.  The warps first count their digits with shared-memory atomics, so
// that the tile's counts are published before the ranking: the look-back of the
// tiles behind it then runs while they rank.  Each warp ranks its items in their order
// (round j: items 32 j .. 32 j + 31) from the lanes of equal digit (one ballot per
// digit bit) and the running position of the digit in the tile, and places them in
// digit order in shared memory; the tile is written in digit runs, so the global
// stores are coalesced.  INDEX: the values are the items' indices (vals_in is not
// read).  DROP: see radix_hist_kernel.
template <class Keys, int ITEMS, int BITS, bool INDEX, bool DROP, bool KEYS_OUT>
__global__ void __launch_bounds__(kRadixThreads, kRadixBlocks) radix_pass_kernel(
    const Keys keys_in, const uint32_t* __restrict__ vals_in, uint32_t* __restrict__ keys_out,
    uint32_t* __restrict__ vals_out, uint32_t n, const uint32_t* __restrict__ d_n, int shift,
    const uint32_t* __restrict__ base, uint32_t* words, uint32_t* next_tile) {
  constexpr int TILE = kRadixThreads * ITEMS;
  constexpr int R = 1 << BITS, PER = (R + kRadixThreads - 1) / kRadixThreads;
  __shared__ uint32_t whist[kRadixWarps][R];
  __shared__ uint32_t gofs[R];  // global position minus tile position of each digit's run
  __shared__ uint32_t s_w[kRadixWarps];
  __shared__ uint32_t sk[TILE], sv[TILE];
  __shared__ uint32_t s_tile, s_items;
  __shared__ int s_gave_up;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_tile = atomicAdd(next_tile, 1u);
    s_gave_up = 0;
  }
  for (int i = lane; i < R; i += 32) whist[warp][i] = 0;
  if (d_n) n = min(n, *d_n);
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint64_t first = (uint64_t)tile * TILE;
  if (first >= n) return;  // capacity launches: no tile after this one waits for it
  const uint32_t here = (uint32_t)min((uint64_t)TILE, n - first);
  const uint32_t slice = (uint32_t)warp * 32 * ITEMS + lane;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t key[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t k = slice + j * 32;
    key[j] = k < here ? keys_in((uint32_t)first + k) : 0xffffffffu;
  }
  auto valid = [&](int j) { return slice + j * 32 < here && (!DROP || key[j] != 0xffffffffu); };
#pragma unroll
  for (int j = 0; j < ITEMS; ++j)
    if (valid(j)) atomicAdd(&whist[warp][(key[j] >> shift) & (R - 1)], 1u);
  uint32_t val[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t k = slice + j * 32;
    val[j] = INDEX ? (uint32_t)first + k : k < here ? vals_in[first + k] : 0u;
  }
  __syncthreads();
  // per digit: the tile's count, and the tile position of each warp's first item
  uint32_t cnt[PER], e;
  {
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int d = threadIdx.x * PER + k;
      cnt[k] = 0;
      if (d < R) {
        uint32_t c = 0;
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) c += whist[w][d];
        cnt[k] = c;
        store_word(words + (size_t)tile * R + d, tile == 0 ? total_word(c) : count_word(c));
      }
    }
    e = block_exclusive<PER>(cnt, s_w);
    uint32_t pos = e;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int d = threadIdx.x * PER + k;
      if (d < R) {
#pragma unroll
        for (int w = 0; w < kRadixWarps; ++w) {
          const uint32_t x = whist[w][d];
          whist[w][d] = pos;
          pos += x;
        }
      }
    }
    if (threadIdx.x == kRadixThreads - 1) s_items = pos;  // items of the tile
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const uint32_t d = (key[j] >> shift) & (R - 1);
    unsigned peers = DROP ? __ballot_sync(kFull, valid(j)) : kFull;
#pragma unroll
    for (int b = 0; b < BITS; ++b) {
      const unsigned bal = __ballot_sync(kFull, (d >> b) & 1u);
      peers &= bal ^ (((d >> b) & 1u) - 1u);
    }
    // (an item past the end has the highest digit and comes last: it moves no other)
    const int before = __popc(peers & lt);
    const uint32_t run = whist[warp][d];
    __syncwarp();
    if (valid(j)) {
      if (before == 0) whist[warp][d] = run + __popc(peers);
      sk[run + before] = key[j];
      sv[run + before] = val[j];
    }
    __syncwarp();
  }
  uint32_t excl[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int d = threadIdx.x * PER + k;
    excl[k] = 0;
    if (d < R && !look_back<R>(words + d, tile, &excl[k])) s_gave_up = 1;
  }
  __syncthreads();
  if (s_gave_up) {  // count the digits of the earlier keys instead of waiting for their tiles
    uint32_t* h = &whist[0][0];
    for (int i = threadIdx.x; i < R; i += kRadixThreads) h[i] = 0;
    __syncthreads();
    for (uint64_t i = threadIdx.x; i < first; i += kRadixThreads) {
      const uint32_t k = keys_in((uint32_t)i);
      if (!DROP || k != 0xffffffffu) atomicAdd(&h[(k >> shift) & (R - 1)], 1u);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PER; ++k) {
      const int d = threadIdx.x * PER + k;
      if (d < R) excl[k] = h[d];
    }
  }
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int d = threadIdx.x * PER + k;
    if (d < R) {
      if (tile) store_word(words + (size_t)tile * R + d, total_word(excl[k] + cnt[k]));
      gofs[d] = base[d] + excl[k] - e;
    }
    e += cnt[k];
  }
  __syncthreads();
  const uint32_t n_out = DROP ? s_items : here;
  for (uint32_t i = threadIdx.x; i < n_out; i += kRadixThreads) {
    const uint32_t k = sk[i];
    const uint32_t pos = gofs[(k >> shift) & (R - 1)] + i;
    if (KEYS_OUT) keys_out[pos] = k;
    vals_out[pos] = sv[i];
  }
}

// ------------------------------------------------------------------ binning helpers
constexpr int kThreads = 256;

__device__ __forceinline__ int row_count(const RowRuns& rr) {
  return max(0, rr.a1 - rr.a0 + 1) + max(0, rr.b1 - rr.b0 + 1);
}

// What a lane knows of its record for the rows of that record that other lanes
// of its warp evaluate: the support conic, the candidate tile rectangle and the view.
struct RowOwner {
  SupportConic k;
  int4 rc;
  int tile_offset, tiles_x, W, H;
};

// The candidate tile rows of the warp's 32 records, flattened over the lanes: f(ri, ty) runs
// for 32 rows at a time, row ty of record ri, in record order and within a record from top to
// bottom, so records with many rows do not leave the lanes of small ones idle.  Every lane
// calls f (it may use warp collectives); ri is -1 for a lane without a row.
// nrows: the rows of this lane's record (0 for none); s_own[lane] must hold it.
template <class F>
__device__ __forceinline__ void for_warp_rows(int nrows, int lane, int* s_incl, const RowOwner* s_own, F f) {
  const int incl = warp_inclusive_scan<int>(nrows, lane);
  s_incl[lane] = incl;
  const int total = __shfl_sync(kFull, incl, 31);
  __syncwarp();
  for (int q0 = 0; q0 < total; q0 += 32) {
    const int q = q0 + lane;
    int ri = -1, ty = 0;
    if (q < total) {
      int lo = 0, hi = 31;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_incl[mid] > q) hi = mid; else lo = mid + 1;
      }
      ri = lo;
      ty = s_own[lo].rc.y + (q - (lo > 0 ? s_incl[lo - 1] : 0));
    }
    f(ri, ty);
  }
  __syncwarp();
}

// Work units of the binning: runs of per_unit consecutive entries of the depth order, one
// warp each.  The counting kernel leaves every unit's first pair position and the writing
// kernel walks the same units with a running position: no scan over the entries, no 64-bit
// offset per entry.  Units are small (the entries nearest to the cameras reach hundreds of
// tiles each: 128 entries per unit instead of 32 made the binning of 500k surfels x 16 views
// 12 % slower), so their totals are scanned in two levels.
constexpr uint32_t kMaxUnits = 65536;
constexpr int kUnitWarps = kThreads / 32;  // units per counting block

// base [units + blocks]: each unit's first position within its counting block, then (from
// units on) each block's first position; first position of a unit = the sum of both.  The last
// block to finish scans the blocks' totals and writes their sum to *total (and, with n32,
// its clamp to cap, raising the capacity bit of *status where it does not fit).
struct UnitTotals {
  uint64_t* base;
  uint32_t* done;   // zeroed
  uint64_t* total;
  uint32_t* n32;
  uint32_t cap;
  int* status;
};

__device__ __forceinline__ uint64_t unit_start(const uint64_t* __restrict__ base, uint32_t units, uint32_t unit) {
  return base[unit] + base[units + unit / kUnitWarps];
}

// sum: this lane's share of its warp's unit (0 for a warp without one); all threads of the block
__device__ __forceinline__ void finish_units(const UnitTotals& t, uint32_t units, uint64_t sum) {
  __shared__ uint64_t s_w[kUnitWarps];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
  if (lane == 0) s_w[warp] = sum;
  __syncthreads();
  const uint32_t unit = blockIdx.x * kUnitWarps + threadIdx.x;
  if (threadIdx.x < kUnitWarps && unit < units) {
    uint64_t e = 0;
    for (int w = 0; w < (int)threadIdx.x; ++w) e += s_w[w];
    t.base[unit] = e;
  }
  if (threadIdx.x == 0) {
    uint64_t c = 0;
    for (int w = 0; w < kUnitWarps; ++w) c += s_w[w];
    t.base[units + blockIdx.x] = c;
    __threadfence();
    s_last = atomicAdd(t.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  uint64_t* blocks = t.base + units;
  const uint32_t per = (gridDim.x + kThreads - 1) / kThreads;
  const uint32_t b0 = min(gridDim.x, threadIdx.x * per), b1 = min(gridDim.x, b0 + per);
  uint64_t mine = 0;
#pragma unroll 8
  for (uint32_t b = b0; b < b1; ++b) mine += __ldcg(blocks + b);
  const uint64_t inc = warp_inclusive_scan<uint64_t>(mine, lane);
  if (lane == 31) s_w[warp] = inc;
  __syncthreads();
  uint64_t run = inc - mine;
  for (int w = 0; w < warp; ++w) run += s_w[w];
#pragma unroll 8
  for (uint32_t b = b0; b < b1; ++b) {
    const uint64_t c = __ldcg(blocks + b);
    blocks[b] = run;
    run += c;
  }
  if (threadIdx.x == kThreads - 1) {
    *t.total = run;
    if (t.n32) {
      *t.n32 = (uint32_t)min(run, (uint64_t)t.cap);
      if (run > (uint64_t)t.cap) atomicOr(t.status, kStatusCapacity);
    }
  }
}

// This lane's record of a round of 32 entries: publishes it in s_own and returns its
// candidate rows (0 without a screen box).
__device__ __forceinline__ int publish_record(uint32_t r, const float4* __restrict__ bin,
                                              const DevCam* __restrict__ cams, int64_t n_gauss, RowOwner* own) {
  const BinView b = load_bin(bin, r);
  if (b.rc.z < b.rc.x) return 0;
  const DevCam& cam = cams[view_of_record(r, n_gauss)];
  *own = RowOwner{support_conic(b.g0, b.g1, b.g2, b.rb), b.rc, cam.tile_offset, cam.tiles_x, cam.W, cam.H};
  return b.rc.w - b.rc.y + 1;
}

// Pairs of the first n entries of the depth order (at most *d_n, the valid ones): one
// closed-form coverage computation per candidate tile row, the rows of a warp's 32 records
// spread over its lanes.
__global__ void __launch_bounds__(kThreads) bin_count_kernel(const uint32_t* __restrict__ order, uint32_t n,
                                                             const uint32_t* __restrict__ d_n, uint32_t per_unit,
                                                             uint32_t units, const float4* __restrict__ bin,
                                                             const DevCam* __restrict__ cams, int64_t n_gauss, int tw,
                                                             int th, const UnitTotals totals) {
  __shared__ RowOwner s_own[kUnitWarps][32];
  __shared__ int s_incl[kUnitWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t unit = blockIdx.x * kUnitWarps + warp;
  n = min(n, *d_n);
  uint64_t sum = 0;
  if (unit < units) {
    for (uint32_t k = 0; k < per_unit; k += 32) {
      const uint64_t i = (uint64_t)unit * per_unit + k + lane;
      if (__all_sync(kFull, i >= n)) break;
      const int nrows = i < n ? publish_record(order[i], bin, cams, n_gauss, &s_own[warp][lane]) : 0;
      for_warp_rows(nrows, lane, s_incl[warp], s_own[warp], [&](int ri, int ty) {
        if (ri < 0) return;
        const RowOwner& o = s_own[warp][ri];
        sum += (uint64_t)row_count(row_runs(o.k, ty, tw, th, o.W, o.H, o.rc));
      });
    }
  }
  finish_units(totals, units, sum);
}

// A row's pairs are written by its own lane where there are few of them, by the whole warp
// above this many.
constexpr int kLongRow = 24;

// Two runs of consecutive values: x_j = a + j for j < la, b + j for la <= j < c.
struct RowItems {
  int la, c;
  uint32_t a, b;
};
__device__ __forceinline__ RowItems row_items(uint32_t a, int la, uint32_t b, int lb) {
  return RowItems{la, la + lb, a, b - (uint32_t)la};
}

// Writes the pairs of one row per lane, (tile(x_j), r) for its c items, from pos on; pairs at
// or past n_pairs are dropped.  Consecutive lanes' pairs are adjacent, so the stores of a
// warp fall into a few neighbouring lines.
template <class T>
__device__ __forceinline__ void write_rows(const RowItems& it, uint64_t pos, uint32_t r, uint32_t n_pairs, int lane,
                                           uint32_t* __restrict__ keys, uint32_t* __restrict__ vals, T tile) {
  const bool is_long = it.c > kLongRow;
  if (!is_long) {
    for (int j = 0; j < it.c; ++j)
      if (pos + (uint64_t)j < (uint64_t)n_pairs) {
        keys[pos + j] = tile((j < it.la ? it.a : it.b) + (uint32_t)j);
        vals[pos + j] = r;
      }
  }
  unsigned left = __ballot_sync(kFull, is_long);
  while (left) {
    const int src = __ffs(left) - 1;
    left &= left - 1u;
    const RowItems o{__shfl_sync(kFull, it.la, src), __shfl_sync(kFull, it.c, src), __shfl_sync(kFull, it.a, src),
                     __shfl_sync(kFull, it.b, src)};
    const uint64_t p = __shfl_sync(kFull, pos, src);
    const uint32_t rr = __shfl_sync(kFull, r, src);
    for (int j = lane; j < o.c; j += 32)
      if (p + (uint64_t)j < (uint64_t)n_pairs) {
        keys[p + j] = tile((j < o.la ? o.a : o.b) + (uint32_t)j);
        vals[p + j] = rr;
      }
  }
}

// The (tile, record) pairs in depth order, entry by entry, rows in order and tiles left to
// right.  The rows of a warp's 32 records come 32 at a time in exactly that order, so a warp
// scan of their tile counts gives every row its position and each lane writes its row: no
// per-entry counts, no search for a pair's row.  What bounds it: the row coverage (ALU) and
// the scattered stores.  500k surfels x 16 views, 18.6 M pairs: 231 -> 118 us against a
// search for every pair's entry and row.
constexpr int kDupThreads = 256;
constexpr int kDupWarps = kDupThreads / 32;

__global__ void __launch_bounds__(kDupThreads) duplicate_kernel(
    const uint32_t* __restrict__ order, uint32_t n, const uint32_t* __restrict__ d_n, uint32_t per_unit,
    uint32_t units, const uint64_t* __restrict__ unit_base, const float4* __restrict__ bin,
    const DevCam* __restrict__ cams, int64_t n_gauss, int tw, int th, uint32_t n_pairs, uint32_t* __restrict__ keys,
    uint32_t* __restrict__ vals) {
  __shared__ RowOwner s_own[kDupWarps][32];
  __shared__ int s_incl[kDupWarps][32];
  __shared__ uint32_t s_rec[kDupWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t unit = blockIdx.x * kDupWarps + warp;
  if (unit >= units) return;
  n = min(n, *d_n);
  uint64_t run = unit_start(unit_base, units, unit);
  for (uint32_t k = 0; k < per_unit; k += 32) {
    const uint64_t i = (uint64_t)unit * per_unit + k + lane;
    if (__all_sync(kFull, i >= n) || run >= (uint64_t)n_pairs) break;
    int nrows = 0;
    if (i < n) {
      const uint32_t r = order[i];
      s_rec[warp][lane] = r;
      nrows = publish_record(r, bin, cams, n_gauss, &s_own[warp][lane]);
    }
    for_warp_rows(nrows, lane, s_incl[warp], s_own[warp], [&](int ri, int ty) {
      RowRuns rr{1, 0, 1, 0};
      uint32_t rowbase = 0, r = 0;
      if (ri >= 0) {
        const RowOwner& o = s_own[warp][ri];
        rr = row_runs(o.k, ty, tw, th, o.W, o.H, o.rc);
        rowbase = (uint32_t)(o.tile_offset + ty * o.tiles_x);
        r = s_rec[warp][ri];
      }
      const RowItems it = row_items(rowbase + (uint32_t)rr.a0, max(0, rr.a1 - rr.a0 + 1), rowbase + (uint32_t)rr.b0,
                                    max(0, rr.b1 - rr.b0 + 1));
      const int inc = warp_inclusive_scan<int>(it.c, lane);
      write_rows(it, run + (uint64_t)(inc - it.c), r, n_pairs, lane, keys, vals, [](uint32_t x) { return x; });
      run += (uint64_t)__shfl_sync(kFull, inc, 31);
    });
  }
}

// [start, end) of every tile in the sorted keys: each thread takes 4
// consecutive keys with one 16-byte load and finds their neighbours across
// lanes with shuffles (the warp's two outer neighbours come from memory).
__global__ void tile_ranges_kernel(const uint32_t* __restrict__ keys, uint32_t n, uint2* __restrict__ ranges,
                                   const uint32_t* __restrict__ d_n) {
  if (d_n) n = min(n, *d_n);
  const int lane = threadIdx.x & 31;
  const uint32_t groups = (n + 3) / 4;
  for (uint32_t base = blockIdx.x * blockDim.x; base < groups; base += gridDim.x * blockDim.x) {
    const uint32_t i0 = (base + threadIdx.x) * 4;
    uint32_t k[4];
    if (i0 + 3 < n) {
      const uint4 v = *reinterpret_cast<const uint4*>(keys + i0);
      k[0] = v.x; k[1] = v.y; k[2] = v.z; k[3] = v.w;
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) k[j] = i0 + j < n ? keys[i0 + j] : 0xffffffffu;
    }
    uint32_t prev = __shfl_up_sync(kFull, k[3], 1);
    uint32_t next = __shfl_down_sync(kFull, k[0], 1);
    if (lane == 0 && i0 > 0 && i0 <= n) prev = keys[i0 - 1];
    if (lane == 31 && i0 + 4 < n) next = keys[i0 + 4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint32_t idx = i0 + j;
      if (idx < n) {
        const uint32_t p = j ? k[j - 1] : prev;
        const uint32_t q = j < 3 ? k[j + 1] : next;
        if (idx == 0 || p != k[j]) ranges[k[j]].x = idx;
        if (idx == n - 1 || q != k[j]) ranges[k[j]].y = idx + 1;
      }
    }
  }
}

}  // namespace

namespace {

// Places of one sort within its scratch (zeroed by the caller): digit positions, counters,
// look-back words.  The scratch may be that of a larger sort; one that is too small is refused
// before any launch.
struct RadixPlaces {
  uint32_t *base, *done, *next_tile, *words;
  size_t tiles;
};
cudaError_t radix_places(const Scratch& scratch, uint32_t n, int passes, int bits, RadixPlaces* w) {
  if (bytes_used(n, passes, bits) > scratch.bytes) return cudaErrorInvalidValue;
  w->tiles = tile_count(n);
  w->base = reinterpret_cast<uint32_t*>(scratch.p);
  w->done = w->base + ((size_t)passes << bits);
  w->next_tile = w->done + 1;
  w->words = w->done + kCounterWords;
  return cudaSuccess;
}

template <class Keys, int BITS, int PASSES, bool DROP>
cudaError_t launch_hist(const Keys& k, uint32_t n, const uint32_t* d_n, const RadixPlaces& w, uint32_t* n_valid,
                        cudaStream_t s) {
  // at least four keys per thread, at most four blocks per SM
  const size_t per_block = 4 * kRadixThreads;
  const uint32_t blocks = (uint32_t)std::min<size_t>((size_t)152 * 4, ((size_t)n + per_block - 1) / per_block);
  radix_hist_kernel<Keys, BITS, PASSES, DROP><<<blocks, kRadixThreads, 0, s>>>(k, n, d_n, w.base, w.done, n_valid);
  return launched();
}

template <class Keys, int BITS, bool INDEX, bool DROP, bool KEYS_OUT>
cudaError_t launch_pass(const Keys& k, const uint32_t* vals, uint32_t* keys_out, uint32_t* vals_out, uint32_t n,
                        const uint32_t* d_n, int p, const RadixPlaces& w, cudaStream_t s) {
  auto pass = n <= kSmallSort ? radix_pass_kernel<Keys, kSmallItems, BITS, INDEX, DROP, KEYS_OUT>
                              : radix_pass_kernel<Keys, kRadixItems, BITS, INDEX, DROP, KEYS_OUT>;
  pass<<<(unsigned)w.tiles, kRadixThreads, 0, s>>>(k, vals, keys_out, vals_out, n, d_n, p * BITS,
                                                   w.base + (size_t)p * (1 << BITS),
                                                   w.words + (size_t)p * w.tiles * (1 << BITS), w.next_tile + p);
  return launched();
}

template <int BITS, int PASSES>
cudaError_t sort_passes(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, uint32_t n,
                        const Scratch& scratch, cudaStream_t s, const uint32_t* d_n) {
  RadixPlaces w;
  cudaError_t e = radix_places(scratch, n, PASSES, BITS, &w);
  if (e == cudaSuccess) e = launch_hist<ArrayKeys, BITS, PASSES, false>(ArrayKeys{keys}, n, d_n, w, nullptr, s);
  uint32_t *kin = keys, *vin = vals, *kout = keys_alt, *vout = vals_alt;
  for (int p = 0; p < PASSES && e == cudaSuccess; ++p) {
    e = launch_pass<ArrayKeys, BITS, false, false, true>(ArrayKeys{kin}, vin, kout, vout, n, d_n, p, w, s);
    std::swap(kin, kout);
    std::swap(vin, vout);
  }
  return e;
}

// The sort of each key width by its digit plan: every width from N to 32 bits is built, so no
// plan is without its kernels.
template <int N>
cudaError_t sort_width(int n_bits, uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, uint32_t n,
                       const Scratch& scratch, cudaStream_t s, const uint32_t* d_n) {
  constexpr DigitPlan plan = digit_plan(N);
  static_assert(plan.bits <= kMaxDigit && plan.bits * plan.passes >= N, "digits of the key");
  if (n_bits == N) return sort_passes<plan.bits, plan.passes>(keys, vals, keys_alt, vals_alt, n, scratch, s, d_n);
  if constexpr (N < 32) return sort_width<N + 1>(n_bits, keys, vals, keys_alt, vals_alt, n, scratch, s, d_n);
  return cudaErrorInvalidValue;
}

}  // namespace

size_t radix_scratch_bytes(uint32_t n, int n_bits) {
  if (n <= 1 || n_bits <= 0) return 16;
  const DigitPlan pl = digit_plan(n_bits);
  return bytes_for(n, pl.passes, pl.bits);
}

bool radix_result_in_alt(uint32_t n, int n_bits) {
  return n > 1 && n_bits > 0 && digit_plan(n_bits).passes % 2 != 0;
}

cudaError_t radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt, uint32_t* vals_alt, uint32_t n,
                             int n_bits, const Scratch& scratch, cudaStream_t s, const uint32_t* d_n) {
  if (n <= 1 || n_bits <= 0) return cudaSuccess;
  return sort_width<1>(n_bits, keys, vals, keys_alt, vals_alt, n, scratch, s, d_n);
}

size_t depth_sort_scratch_bytes(uint32_t n) { return bytes_for(n, 4, 8); }

cudaError_t depth_sort(uint32_t* keys, uint32_t* keys_alt, uint32_t* order, uint32_t* order_alt, uint32_t n,
                       uint32_t* n_valid, const Scratch& scratch, cudaStream_t s) {
  if (n == 0) return cudaMemsetAsync(n_valid, 0, sizeof(uint32_t), s);
  RadixPlaces w;
  cudaError_t e = radix_places(scratch, n, 4, 8, &w);
  if (e == cudaSuccess) e = launch_hist<ArrayKeys, 8, 4, true>(ArrayKeys{keys}, n, nullptr, w, n_valid, s);
  if (e == cudaSuccess)  // the first pass makes the indices and leaves the culled records out
    e = launch_pass<ArrayKeys, 8, true, true, true>(ArrayKeys{keys}, nullptr, keys_alt, order_alt, n, nullptr, 0, w, s);
  if (e == cudaSuccess)
    e = launch_pass<ArrayKeys, 8, false, false, true>(ArrayKeys{keys_alt}, order_alt, keys, order, n, n_valid, 1, w, s);
  if (e == cudaSuccess)
    e = launch_pass<ArrayKeys, 8, false, false, true>(ArrayKeys{keys}, order, keys_alt, order_alt, n, n_valid, 2, w, s);
  if (e == cudaSuccess)
    e = launch_pass<ArrayKeys, 8, false, false, false>(ArrayKeys{keys_alt}, order_alt, nullptr, order, n, n_valid, 3,
                                                       w, s);
  return e;
}

size_t tile_order_scratch_bytes(uint32_t n_tiles) { return bytes_for(n_tiles, 1, 4); }

cudaError_t launch_tile_order(const uint2* ranges, const uint2* ranges2, uint32_t n_tiles, uint32_t* ids,
                              const Scratch& scratch, cudaStream_t s, const uint32_t** n_nonempty) {
  RadixPlaces w;
  cudaError_t e = radix_places(scratch, n_tiles, 1, 4, &w);
  if (e != cudaSuccess) return e;
  if (n_nonempty) *n_nonempty = w.base + 15;  // first position of the empty tiles' class
  if (n_tiles == 0) return cudaSuccess;
  const QueueKeys k{ranges, ranges2};
  e = launch_hist<QueueKeys, 4, 1, false>(k, n_tiles, nullptr, w, nullptr, s);
  if (e != cudaSuccess) return e;
  return launch_pass<QueueKeys, 4, true, false, false>(k, nullptr, nullptr, ids, n_tiles, nullptr, 0, w, s);
}

cudaError_t launch_tile_ranges(const uint32_t* keys, uint32_t n_pairs, uint2* ranges, cudaStream_t s,
                               const uint32_t* d_n) {
  if (n_pairs == 0) return cudaSuccess;
  const uint32_t blocks = (n_pairs / 4 + 256) / 256;
  tile_ranges_kernel<<<blocks < 152u * 16u ? blocks : 152u * 16u, 256, 0, s>>>(keys, n_pairs, ranges, d_n);
  return launched();
}

}  // namespace ocgs

// ------------------------------------------------------------------ two-pass binning
// The first pass bins only the records at the front of the depth order; the
// tiles whose pixels all stop inside that prefix (the front-to-back walk of
// Sec. 4.3 ends when T falls below its bound) are final.  The second pass bins
// the records behind the front, but only into the tiles still open, and those
// tiles continue from where the first pass stopped.  Each tile's list is the
// one a single pass builds (records in depth order), split in two segments.
namespace ocgs {
namespace {

__device__ __forceinline__ int4 bin_rect(const float4 b2) {
  const uint32_t xy = __float_as_uint(b2.z), zw = __float_as_uint(b2.w);
  return make_int4((int)(int16_t)(xy & 0xffffu), (int)(int16_t)(xy >> 16), (int)(int16_t)(zw & 0xffffu),
                   (int)(int16_t)(zw >> 16));
}

// open tiles among [rowbase + x0, rowbase + x1] from the exclusive prefix P of the open flags
__device__ __forceinline__ int open_in(const uint32_t* __restrict__ P, uint32_t rowbase, int x0, int x1) {
  return x1 < x0 ? 0 : (int)(P[rowbase + (uint32_t)x1 + 1u] - P[rowbase + (uint32_t)x0]);
}

// The exclusive prefix P [n + 1] of the open flags and the open tiles in ascending order
// (open_ids[P[t]] = t for every open tile t), in one kernel: a block scans its tile of
// kScanTile flags and adds the totals of the tiles before it, found by the look-back of the
// sorts (a wait that is given up counts the earlier flags instead).
constexpr int kScanTile = kThreads * 16;

__global__ void __launch_bounds__(kThreads) open_scan_kernel(const uint32_t* __restrict__ open, uint32_t n,
                                                             uint32_t* __restrict__ P, uint32_t* __restrict__ open_ids,
                                                             uint32_t* words, uint32_t* next_tile) {
  static_assert(kScanTile <= kMaxTileCount, "look-back words");
  constexpr int kItems16 = kScanTile / kThreads;
  __shared__ uint32_t s_w[kThreads / 32];
  __shared__ uint32_t s_tile, s_excl;
  __shared__ int s_gave_up;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    s_tile = atomicAdd(next_tile, 1u);
    s_gave_up = 0;
  }
  __syncthreads();
  const uint32_t tile = s_tile, first = tile * (uint32_t)kScanTile;
  const uint32_t wbase = first + (uint32_t)warp * 32 * kItems16 + lane;
  uint32_t f[kItems16], pre[kItems16];
  uint32_t run = 0;  // open flags of this warp's earlier rounds
#pragma unroll
  for (int j = 0; j < kItems16; ++j) f[j] = wbase + j * 32 < n ? open[wbase + j * 32] : 0u;
#pragma unroll
  for (int j = 0; j < kItems16; ++j) {
    const unsigned m = __ballot_sync(kFull, f[j] != 0u);
    pre[j] = run + (uint32_t)__popc(m & ((1u << lane) - 1u));
    run += (uint32_t)__popc(m);
  }
  if (lane == 0) s_w[warp] = run;
  __syncthreads();
  uint32_t off = 0, total = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) {
    off += w < warp ? s_w[w] : 0u;
    total += s_w[w];
  }
  if (warp == 0) {
    if (lane == 0) store_word(words + tile, tile == 0 ? total_word(total) : count_word(total));
    uint32_t e = 0;
    const bool found = look_back_warp(words, tile, lane, &e);
    if (lane == 0) {
      if (!found) s_gave_up = 1;
      s_excl = e;
    }
  }
  __syncthreads();
  if (s_gave_up) {
    if (threadIdx.x == 0) s_excl = 0;
    __syncthreads();
    uint32_t c = 0;
    for (uint32_t i = threadIdx.x; i < first; i += kThreads) c += open[i] ? 1u : 0u;
    atomicAdd(&s_excl, c);
    __syncthreads();
  }
  const uint32_t excl = s_excl;
  if (threadIdx.x == 0) {
    if (tile) store_word(words + tile, total_word(excl + total));
    if (first + (uint32_t)kScanTile >= n) P[n] = excl + total;
  }
#pragma unroll
  for (int j = 0; j < kItems16; ++j) {
    const uint32_t t = wbase + j * 32;
    if (t < n) {
      const uint32_t q = excl + off + pre[j];
      P[t] = q;
      if (f[j]) open_ids[q] = t;
    }
  }
}

// Second pass, candidates and counts: a unit's warp tests its entries (records behind the
// front, in depth order) for an open tile in their screen box (row sums of the open flags
// from their prefix P) and collects the few that have one; every 32 of those, their exact
// open tiles are counted with the rows spread over the lanes.  The unit's candidates and
// their counts stay in its own stretch [unit * per_unit, ...) of cand and counts, in order,
// and n_cand[unit] holds their number: nothing is compacted over the whole list.
__global__ void __launch_bounds__(kThreads) open_count_kernel(const uint32_t* __restrict__ order, uint32_t n,
                                                              uint32_t per_unit, uint32_t units,
                                                              const float4* __restrict__ bin,
                                                              const DevCam* __restrict__ cams, int64_t n_gauss, int tw,
                                                              int th, const uint32_t* __restrict__ P,
                                                              uint32_t* __restrict__ cand,
                                                              uint32_t* __restrict__ counts,
                                                              uint32_t* __restrict__ n_cand, const UnitTotals totals) {
  __shared__ RowOwner s_own[kUnitWarps][32];
  __shared__ int s_incl[kUnitWarps][32], s_cnt[kUnitWarps][32];
  __shared__ uint32_t s_queue[kUnitWarps][64];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t unit = blockIdx.x * kUnitWarps + warp;
  uint64_t sum = 0;
  if (unit < units) {
    const uint64_t base = (uint64_t)unit * per_unit;
    uint32_t* queue = s_queue[warp];
    uint32_t waiting = 0, found = 0;
    auto count = [&](uint32_t m) {  // the first m <= 32 waiting candidates
      int nrows = 0;
      if (lane < (int)m) {
        const uint32_t r = queue[lane];
        nrows = publish_record(r, bin, cams, n_gauss, &s_own[warp][lane]);
        cand[base + found + lane] = r;
      }
      s_cnt[warp][lane] = 0;
      for_warp_rows(nrows, lane, s_incl[warp], s_own[warp], [&](int ri, int ty) {
        if (ri < 0) return;
        const RowOwner& o = s_own[warp][ri];
        const RowRuns rr = row_runs(o.k, ty, tw, th, o.W, o.H, o.rc);
        const uint32_t rowbase = (uint32_t)(o.tile_offset + ty * o.tiles_x);
        const int c = open_in(P, rowbase, rr.a0, rr.a1) + open_in(P, rowbase, rr.b0, rr.b1);
        if (c) atomicAdd(&s_cnt[warp][ri], c);
      });
      if (lane < (int)m) {
        counts[base + found + lane] = (uint32_t)s_cnt[warp][lane];
        sum += (uint64_t)s_cnt[warp][lane];
      }
      found += m;
      __syncwarp();
    };
    for (uint32_t k = 0; k < per_unit; k += 32) {
      const uint64_t i = base + k + lane;
      if (__all_sync(kFull, i >= n)) break;
      uint32_t r = 0;
      bool open_here = false;
      if (i < n) {
        r = order[i];
        const int4 rc = bin_rect(bin[3 * (size_t)r + 2]);
        if (rc.z >= rc.x) {
          const DevCam& cam = cams[view_of_record(r, n_gauss)];
          const uint32_t row0 = (uint32_t)(cam.tile_offset + rc.y * cam.tiles_x);
          int c = 0;
          for (int ty = rc.y; ty <= rc.w; ++ty) c += open_in(P, row0 + (uint32_t)((ty - rc.y) * cam.tiles_x), rc.x, rc.z);
          open_here = c > 0;
        }
      }
      const unsigned m = __ballot_sync(kFull, open_here);
      if (open_here) queue[waiting + __popc(m & lt)] = r;
      waiting += (uint32_t)__popc(m);
      __syncwarp();
      if (waiting >= 32) {
        count(32);
        const uint32_t rest = queue[32 + lane];
        __syncwarp();
        queue[lane] = rest;
        waiting -= 32;
        __syncwarp();
      }
    }
    if (waiting) count(waiting);
    if (lane == 0) n_cand[unit] = found;
  }
  finish_units(totals, units, sum);
}

// The open tiles of the run [x0, x1] of a tile row are the contiguous slice
// open_ids[P[rowbase + x0], P[rowbase + x1 + 1]) of the compacted open ids.
struct OpenSlice {
  uint32_t start;
  int count;
};
__device__ __forceinline__ OpenSlice open_slice(const uint32_t* __restrict__ P, uint32_t rowbase, int x0, int x1) {
  if (x1 < x0) return OpenSlice{0u, 0};
  const uint32_t a = P[rowbase + (uint32_t)x0];
  return OpenSlice{a, (int)(P[rowbase + (uint32_t)x1 + 1u] - a)};
}

// The second-pass pairs in depth order, as in duplicate_kernel: each row's open tiles are the
// slices of its two runs.  A block takes the candidates of kUnitWarps units together: it
// scans their counts, and its warps take 32 candidates at a time, so that the lanes are full
// although a unit holds few candidates and the block's units hold unequal numbers.
constexpr int kGroup = kDupThreads * 4;  // candidates of a block per round

__global__ void __launch_bounds__(kDupThreads) duplicate_open_kernel(
    const uint32_t* __restrict__ cand, const uint32_t* __restrict__ counts, const uint32_t* __restrict__ n_cand,
    uint32_t per_unit, uint32_t units, const uint64_t* __restrict__ unit_base, const float4* __restrict__ bin,
    const DevCam* __restrict__ cams, int64_t n_gauss, int tw, int th, const uint32_t* __restrict__ open_ids,
    const uint32_t* __restrict__ P, uint32_t n_pairs, uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  __shared__ RowOwner s_own[kDupWarps][32];
  __shared__ int s_incl[kDupWarps][32];
  __shared__ uint32_t s_first[kUnitWarps + 1];  // first candidate of each unit within the block's list
  __shared__ uint32_t s_rec[kGroup], s_pos[kGroup], s_w[kDupWarps];
  static_assert(kDupWarps == kUnitWarps, "one block per counting block");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t u0 = blockIdx.x * kUnitWarps;
  if (threadIdx.x == 0) {
    uint32_t c = 0;
    for (int u = 0; u < kUnitWarps; ++u) {
      s_first[u] = c;
      if (u0 + u < units) c += n_cand[u0 + u];
    }
    s_first[kUnitWarps] = c;
  }
  __syncthreads();
  const uint32_t found = s_first[kUnitWarps];
  uint64_t start = unit_start(unit_base, units, u0);  // first pair of the group
  for (uint32_t g0 = 0; g0 < found; g0 += kGroup) {
    const uint32_t here = min((uint32_t)kGroup, found - g0);
    // 4 consecutive candidates per thread
    uint32_t c[4], mine = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t q = threadIdx.x * 4 + k;
      c[k] = 0;
      if (q < here) {
        int u = 0;
#pragma unroll
        for (int v = 1; v < kUnitWarps; ++v) u += s_first[v] <= g0 + q ? 1 : 0;
        const uint64_t at = (uint64_t)(u0 + u) * per_unit + (g0 + q - s_first[u]);
        s_rec[q] = cand[at];
        c[k] = counts[at];
      }
      mine += c[k];
    }
    const uint32_t inc = warp_inclusive_scan<uint32_t>(mine, lane);
    if (lane == 31) s_w[warp] = inc;
    __syncthreads();
    uint32_t before = inc - mine, total = 0;
#pragma unroll
    for (int w = 0; w < kDupWarps; ++w) {
      before += w < warp ? s_w[w] : 0u;
      total += s_w[w];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      s_pos[threadIdx.x * 4 + k] = before;
      before += c[k];
    }
    __syncthreads();
    for (uint32_t q0 = warp * 32; q0 < here; q0 += kDupThreads) {
      const uint32_t q = q0 + lane;
      const int nrows = q < here ? publish_record(s_rec[q], bin, cams, n_gauss, &s_own[warp][lane]) : 0;
      uint64_t run = start + s_pos[q0];
      for_warp_rows(nrows, lane, s_incl[warp], s_own[warp], [&](int ri, int ty) {
        OpenSlice sa{0u, 0}, sb{0u, 0};
        uint32_t r = 0;
        if (ri >= 0) {
          const RowOwner& o = s_own[warp][ri];
          const RowRuns rr = row_runs(o.k, ty, tw, th, o.W, o.H, o.rc);
          const uint32_t rowbase = (uint32_t)(o.tile_offset + ty * o.tiles_x);
          sa = open_slice(P, rowbase, rr.a0, rr.a1);
          sb = open_slice(P, rowbase, rr.b0, rr.b1);
          r = s_rec[q0 + ri];
        }
        const RowItems it = row_items(sa.start, sa.count, sb.start, sb.count);
        const int row_inc = warp_inclusive_scan<int>(it.c, lane);
        write_rows(it, run + (uint64_t)(row_inc - it.c), r, n_pairs, lane, keys, vals,
                   [&](uint32_t x) { return open_ids[x]; });
        run += (uint64_t)__shfl_sync(kFull, row_inc, 31);
      });
    }
    start += total;
    __syncthreads();  // the next group overwrites s_rec, s_pos and s_w
  }
}

struct UnitPlan {
  uint32_t per_unit, units;
};
// Rounds of 32 entries per unit so that there are at most kMaxUnits units.
UnitPlan unit_plan(uint32_t n) {
  const uint32_t per = 32u * std::max(1u, (uint32_t)(((uint64_t)n + 32ull * kMaxUnits - 1) / (32ull * kMaxUnits)));
  return UnitPlan{per, (uint32_t)(((uint64_t)n + per - 1) / per)};
}

}  // namespace

// (the number of units is not monotonic in n)
size_t unit_capacity(uint32_t n) { return std::min<size_t>(((size_t)n + 31) / 32, kMaxUnits); }
size_t unit_base_words(uint32_t n) { return unit_capacity(n) + (unit_capacity(n) + kUnitWarps - 1) / kUnitWarps; }

cudaError_t launch_bin_count(const uint32_t* order, uint32_t n, const uint32_t* d_n, const float4* bin,
                             const DevCam* cams, int64_t n_gauss, int tile_w, int tile_h, uint64_t* unit_base,
                             uint32_t* done, uint64_t* total, cudaStream_t s, uint32_t* n32, uint32_t cap,
                             int* status) {
  if (n == 0) return cudaMemsetAsync(total, 0, sizeof(uint64_t), s);
  const UnitPlan u = unit_plan(n);
  bin_count_kernel<<<(u.units + kUnitWarps - 1) / kUnitWarps, kThreads, 0, s>>>(
      order, n, d_n, u.per_unit, u.units, bin, cams, n_gauss, tile_w, tile_h,
      UnitTotals{unit_base, done, total, n32, cap, status});
  return launched();
}

cudaError_t launch_duplicate(const uint32_t* order, uint32_t n, const uint32_t* d_n, const uint64_t* unit_base,
                             const float4* bin, const DevCam* cams, int64_t n_gauss, int tile_w, int tile_h,
                             uint32_t n_pairs, uint32_t* keys, uint32_t* vals, cudaStream_t s) {
  if (n_pairs == 0 || n == 0) return cudaSuccess;
  const UnitPlan u = unit_plan(n);
  duplicate_kernel<<<(u.units + kDupWarps - 1) / kDupWarps, kDupThreads, 0, s>>>(
      order, n, d_n, u.per_unit, u.units, unit_base, bin, cams, n_gauss, tile_w, tile_h, n_pairs, keys, vals);
  return launched();
}

size_t open_scan_words(uint32_t n_tiles) { return ((size_t)n_tiles + kScanTile - 1) / kScanTile + 1; }

cudaError_t launch_open_scan(const uint32_t* open, uint32_t n_tiles, uint32_t* P, uint32_t* open_ids, uint32_t* words,
                             cudaStream_t s) {
  const uint32_t blocks = (uint32_t)open_scan_words(n_tiles) - 1;
  open_scan_kernel<<<blocks, kThreads, 0, s>>>(open, n_tiles, P, open_ids, words, words + blocks);
  return launched();
}

cudaError_t launch_open_count(const uint32_t* order, uint32_t n, const float4* bin, const DevCam* cams,
                              int64_t n_gauss, int tile_w, int tile_h, const uint32_t* P, uint32_t* cand,
                              uint32_t* counts, uint32_t* n_cand, uint64_t* unit_base, uint32_t* done,
                              uint64_t* total, cudaStream_t s) {
  if (n == 0) return cudaMemsetAsync(total, 0, sizeof(uint64_t), s);
  const UnitPlan u = unit_plan(n);
  open_count_kernel<<<(u.units + kUnitWarps - 1) / kUnitWarps, kThreads, 0, s>>>(
      order, n, u.per_unit, u.units, bin, cams, n_gauss, tile_w, tile_h, P, cand, counts, n_cand,
      UnitTotals{unit_base, done, total, nullptr, 0u, nullptr});
  return launched();
}

cudaError_t launch_duplicate_open(const uint32_t* cand, uint32_t n, const uint32_t* counts, const uint32_t* n_cand,
                                  const uint64_t* unit_base, const float4* bin, const DevCam* cams, int64_t n_gauss,
                                  int tile_w, int tile_h, const uint32_t* open_ids, const uint32_t* P,
                                  uint32_t n_pairs, uint32_t* keys, uint32_t* vals, cudaStream_t s) {
  if (n_pairs == 0 || n == 0) return cudaSuccess;
  const UnitPlan u = unit_plan(n);
  duplicate_open_kernel<<<(u.units + kDupWarps - 1) / kDupWarps, kDupThreads, 0, s>>>(
      cand, counts, n_cand, u.per_unit, u.units, unit_base, bin, cams, n_gauss, tile_w, tile_h, open_ids, P, n_pairs,
      keys, vals);
  return launched();
}

}  // namespace ocgs
