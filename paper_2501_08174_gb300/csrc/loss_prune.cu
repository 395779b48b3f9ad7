// Background loss (Eq. 1) with its fused adjoint, and the pruning keep-set
// compaction (Sec. 4.3).
#include "lookback.cuh"
#include "ocgs.h"

#include <cmath>
#include <cstring>
#include <mutex>
#include <type_traits>

namespace ocgs {
namespace {

constexpr int kLossThreads = 256;
constexpr int kLossLoads = 2;  // pixels per thread whose loads are in flight together

// Each block reduces kLossBlockPixels pixels of one view, in a fixed order
// (compensated float32 sums per thread, merged into one FP64 partial per block),
// and a second pass adds the partials of a view in block order, so the loss is
// bitwise reproducible.
__global__ void __launch_bounds__(kLossThreads) bg_loss_partial_kernel(
    const float* __restrict__ alpha, const uint8_t* __restrict__ mask, const DevCam* __restrict__ cams,
    int n_views, const int* __restrict__ block_prefix, float gamma, double* __restrict__ partial,
    float* __restrict__ d_alpha) {
  const int b = blockIdx.x;
  const int v = view_of_tile(block_prefix, n_views, b);
  const DevCam& cam = cams[v];
  const int64_t npix = (int64_t)cam.W * cam.H;
  const int64_t lo = (int64_t)(b - block_prefix[v]) * kLossBlockPixels;
  const int64_t hi = (lo + kLossBlockPixels < npix) ? lo + kLossBlockPixels : npix;
  const float g = gamma / (float)npix;
  CompSum acc[1];
  for (int64_t k0 = lo + threadIdx.x; k0 < hi; k0 += kLossLoads * kLossThreads) {
    float a[kLossLoads], d[kLossLoads];
    bool bg[kLossLoads];
#pragma unroll
    for (int u = 0; u < kLossLoads; ++u) {
      const int64_t k = k0 + u * kLossThreads, p = cam.pix_offset + k;
      bg[u] = k < hi && !mask[p];
      a[u] = k < hi ? alpha[p] : 0.f;
      d[u] = bg[u] && d_alpha ? d_alpha[p] : 0.f;  // (1 - M) adds nothing to the others
    }
#pragma unroll
    for (int u = 0; u < kLossLoads; ++u) {
      acc[0].add(a[u] * (bg[u] ? 1.f : 0.f));  // alpha (1 - M) is exact
      if (bg[u] && d_alpha) d_alpha[cam.pix_offset + k0 + u * kLossThreads] = d[u] + g;
    }
  }
  block_comp_sums<kLossThreads, 1>(acc, partial + b);
}

// Masked L1 (Eq. 2, L1 part): |I M - R M| summed per block, with the adjoint
// weight * sign(R - I) * M / (3 h w) added into d_rgb.  Each difference is
// taken exactly as a float pair (TwoSum: R - I = d + e, |e| <= ulp(d) / 2, so
// |R - I| = |d| + sign(d) e) and summed with compensation, so the loss differs
// from the exact one by rounding far below float precision; the sign of d is
// the sign of the exact difference (d = 0 only when R = I).
__global__ void __launch_bounds__(kLossThreads) l1_partial_kernel(
    const float* __restrict__ rgb, const float* __restrict__ target, const uint8_t* __restrict__ mask,
    const DevCam* __restrict__ cams, int n_views, const int* __restrict__ block_prefix, float weight,
    double* __restrict__ partial, float* __restrict__ d_rgb) {
  const int b = blockIdx.x;
  const int v = view_of_tile(block_prefix, n_views, b);
  const DevCam& cam = cams[v];
  const int64_t npix = (int64_t)cam.W * cam.H;
  const int64_t lo = (int64_t)(b - block_prefix[v]) * kLossBlockPixels;
  const int64_t hi = (lo + kLossBlockPixels < npix) ? lo + kLossBlockPixels : npix;
  const float g = weight / (3.0f * (float)npix);
  CompSum acc[1];
  for (int64_t k0 = lo + threadIdx.x; k0 < hi; k0 += kLossLoads * kLossThreads) {
    bool m[kLossLoads];
    float x[kLossLoads][3], y[kLossLoads][3], q[kLossLoads][3];
#pragma unroll
    for (int u = 0; u < kLossLoads; ++u) {
      const int64_t k = k0 + u * kLossThreads;
      m[u] = k < hi && mask[cam.pix_offset + k];
    }
#pragma unroll
    for (int u = 0; u < kLossLoads; ++u) {
      const int64_t p = cam.pix_offset + k0 + u * kLossThreads;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        x[u][c] = m[u] ? rgb[3 * p + c] : 0.f;
        y[u][c] = m[u] ? target[3 * p + c] : 0.f;
        q[u][c] = m[u] && d_rgb ? d_rgb[3 * p + c] : 0.f;
      }
    }
#pragma unroll
    for (int u = 0; u < kLossLoads; ++u) {
      if (!m[u]) continue;
      const int64_t p = cam.pix_offset + k0 + u * kLossThreads;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        float e;
        const float d = two_sum(x[u][c], -y[u][c], e);
        acc[0].add(fabsf(d), d > 0.f ? e : -e);
        if (d_rgb) d_rgb[3 * p + c] = q[u][c] + (d > 0.f ? g : (d < 0.f ? -g : 0.f));
      }
    }
  }
  block_comp_sums<kLossThreads, 1>(acc, partial + b);
}

// one CTA per view
__global__ void __launch_bounds__(kViewSumThreads) bg_loss_final_kernel(const double* __restrict__ partial,
                                                                       const int* __restrict__ block_prefix,
                                                                       const DevCam* __restrict__ cams, double scale,
                                                                       double* __restrict__ loss) {
  const int v = blockIdx.x;
  double t;
  view_block_sums<1>(partial, block_prefix[v], block_prefix[v + 1], &t);
  if (threadIdx.x == 0) loss[v] = t / ((double)cams[v].W * (double)cams[v].H) * scale;
}

// ----------------------------------------------------------------------------- pruning
using namespace lookback;

constexpr int kPruneThreads = 256;  // Gaussians per block

// Rows list[0 .. kept) of an array of W floats per Gaussian, to the rows from base on: the
// block's kept rows are contiguous in the output, so the stores are coalesced, and each
// source row is read by neighbouring lanes.
template <int W, typename V>
__device__ __forceinline__ void copy_rows_as(const float* __restrict__ in, float* __restrict__ out, int64_t i0,
                                             const uint16_t* list, int kept, int64_t base) {
  constexpr int Q = W * sizeof(float) / sizeof(V);  // vectors per row
  const V* src = reinterpret_cast<const V*>(in) + i0 * Q;
  V* dst = reinterpret_cast<V*>(out) + base * Q;
  constexpr int kBatch = Q >= 4 ? 4 : Q;  // loads in flight per thread
  const int total = kept * Q;
  for (int k0 = threadIdx.x; k0 < total; k0 += kBatch * kPruneThreads) {
    V v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int k = k0 + u * kPruneThreads;
      if (k < total) v[u] = __ldcs(src + ((int)list[k / Q] * Q + k % Q));
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int k = k0 + u * kPruneThreads;
      if (k < total) __stcs(dst + k, v[u]);
    }
  }
}
template <int W>
__device__ __forceinline__ void copy_rows(const float* __restrict__ in, float* __restrict__ out, int64_t i0,
                                          const uint16_t* list, int kept, int64_t base) {
  const uintptr_t both = reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out);
  if (W % 4 == 0 && both % 16 == 0) copy_rows_as<W, typename std::conditional<W % 4 == 0, float4, float>::type>(in, out, i0, list, kept, base);
  else if (W % 2 == 0 && both % 8 == 0) copy_rows_as<W, typename std::conditional<W % 2 == 0, float2, float>::type>(in, out, i0, list, kept, base);
  else copy_rows_as<W, float>(in, out, i0, list, kept, base);
}

__device__ __forceinline__ bool is_kept(float s, float tau) { return s > tau; }
__device__ __forceinline__ bool is_border(float s, float tau) { return fabsf(s - tau) <= 1e-6f; }

// Kept and border counts of every kPruneThreads Gaussians (a tile), one warp each, in two levels:
// tiles[2 t + w] the count (w = 0 kept, 1 border) of the tiles before tile t in its block of
// kPruneWarps, blocks[2 b + w] that of the blocks before block b, which the last block to finish
// fills in; the totals go to n_out.  (With one level the last block walked every tile: 10 M
// Gaussians of degree 0, all kept, took 475 us against 405 with scan kernels over all of them;
// this form, with three of a row's loads in flight in the copy, 315.)
constexpr int kPruneWarps = kPruneThreads / 32;
__global__ void __launch_bounds__(kPruneThreads) prune_count_kernel(const float* __restrict__ score, uint32_t n,
                                                                    float tau, uint32_t n_tiles, uint32_t* tiles,
                                                                    uint32_t* blocks, uint32_t* done,
                                                                    uint32_t* __restrict__ n_out) {
  constexpr int kRounds = kPruneThreads / 32;
  __shared__ uint32_t s_w[2][kPruneWarps];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tile = blockIdx.x * kPruneWarps + warp;
  uint32_t ck = 0, cb = 0;  // NaN is neither kept nor at the border
  if (tile < n_tiles) {
    const int64_t i0 = (int64_t)tile * kPruneThreads + lane;
    float s[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) s[r] = i0 + 32 * r < n ? score[i0 + 32 * r] : __int_as_float(0x7fc00000);
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
      ck += (uint32_t)__popc(__ballot_sync(kFull, is_kept(s[r], tau)));
      cb += (uint32_t)__popc(__ballot_sync(kFull, is_border(s[r], tau)));
    }
  }
  if (lane == 0) {
    s_w[0][warp] = ck;
    s_w[1][warp] = cb;
  }
  __syncthreads();
  if (threadIdx.x < 2 * kPruneWarps) {
    const int t = threadIdx.x >> 1, which = threadIdx.x & 1;
    uint32_t before = 0;
    for (int w = 0; w < t; ++w) before += s_w[which][w];
    if (blockIdx.x * kPruneWarps + t < n_tiles) tiles[2 * (blockIdx.x * kPruneWarps + t) + which] = before;
    if (t == kPruneWarps - 1) blocks[2 * blockIdx.x + which] = before + s_w[which][t];
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint32_t per = (gridDim.x + kPruneThreads - 1) / kPruneThreads;
  const uint32_t b0 = min(gridDim.x, threadIdx.x * per), b1 = min(gridDim.x, b0 + per);
  uint2* both = reinterpret_cast<uint2*>(blocks);  // (kept, border)
  uint2 sum = make_uint2(0u, 0u);
#pragma unroll 8
  for (uint32_t b = b0; b < b1; ++b) {
    const uint2 x = __ldcg(both + b);
    sum.x += x.x;
    sum.y += x.y;
  }
  const uint2 inc = make_uint2(warp_inclusive_scan<uint32_t>(sum.x, lane), warp_inclusive_scan<uint32_t>(sum.y, lane));
  if (lane == 31) {
    s_w[0][warp] = inc.x;
    s_w[1][warp] = inc.y;
  }
  __syncthreads();
  uint2 run = make_uint2(inc.x - sum.x, inc.y - sum.y);
  for (int w = 0; w < warp; ++w) {
    run.x += s_w[0][w];
    run.y += s_w[1][w];
  }
#pragma unroll 8
  for (uint32_t b = b0; b < b1; ++b) {
    const uint2 x = __ldcg(both + b);
    both[b] = run;
    run.x += x.x;
    run.y += x.y;
  }
  if (threadIdx.x == kPruneThreads - 1) {
    n_out[0] = run.x;
    n_out[1] = run.y;
  }
}

// Stable compaction: a block lists its kept Gaussians and copies their rows.
//
// What bounds it: HBM (464 bytes per kept Gaussian of degree 3).  One thread per Gaussian
// copying its 48 coefficients at a stride of 192 bytes took 292 us for 1M Gaussians of which
// 69 % are kept; finding the positions by a look-back inside this kernel 143 us (its blocks
// waited for one another more than they copied); this form 62 us with its count kernel.
template <int DEG>
__global__ void __launch_bounds__(kPruneThreads) prune_copy_kernel(const float* __restrict__ score, uint32_t n,
                                                                   float tau, const GaussPtrs in, GaussOut out,
                                                                   int64_t* __restrict__ border_idx,
                                                                   int64_t border_cap,
                                                                   const uint2* __restrict__ tiles,
                                                                   const uint2* __restrict__ blocks) {
  __shared__ uint16_t s_list[kPruneThreads];
  __shared__ uint32_t s_k[kPruneWarps], s_b[kPruneWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t i0 = (int64_t)blockIdx.x * kPruneThreads, i = i0 + threadIdx.x;
  const uint2 in_block = tiles[blockIdx.x], of_block = blocks[blockIdx.x / kPruneWarps];
  const uint32_t bk = in_block.x + of_block.x, bb = in_block.y + of_block.y;
  const float s = i < n ? score[i] : __int_as_float(0x7fc00000);
  const bool keep = is_kept(s, tau), border = is_border(s, tau);
  const unsigned mk = __ballot_sync(kFull, keep), mb = __ballot_sync(kFull, border);
  if (lane == 0) {
    s_k[warp] = (uint32_t)__popc(mk);
    s_b[warp] = (uint32_t)__popc(mb);
  }
  __syncthreads();
  uint32_t ok = (uint32_t)__popc(mk & lt), ob = (uint32_t)__popc(mb & lt), kept = 0;
#pragma unroll
  for (int w = 0; w < kPruneWarps; ++w) {
    ok += w < warp ? s_k[w] : 0u;
    ob += w < warp ? s_b[w] : 0u;
    kept += s_k[w];
  }
  if (keep) s_list[ok] = (uint16_t)threadIdx.x;
  if (border && border_idx && (int64_t)(bb + ob) < border_cap) border_idx[bb + ob] = i;
  __syncthreads();
  copy_rows<3 * (DEG + 1) * (DEG + 1)>(in.sh, out.sh, i0, s_list, (int)kept, bk);
  copy_rows<4>(in.quat, out.quat, i0, s_list, (int)kept, bk);
  copy_rows<3>(in.xyz, out.xyz, i0, s_list, (int)kept, bk);
  copy_rows<2>(in.scale, out.scale, i0, s_list, (int)kept, bk);
  copy_rows<1>(in.opacity, out.opacity, i0, s_list, (int)kept, bk);
}

}  // namespace

cudaError_t launch_background_loss(const float* alpha, const uint8_t* mask, const DevCam* cams,
                                   int n_views, const int* block_prefix, int n_blocks, float gamma,
                                   double* partial, double* loss, float* d_alpha, cudaStream_t s) {
  if (n_blocks > 0) {
    bg_loss_partial_kernel<<<n_blocks, kLossThreads, 0, s>>>(alpha, mask, cams, n_views, block_prefix,
                                                             gamma, partial, d_alpha);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
  }
  bg_loss_final_kernel<<<n_views, kViewSumThreads, 0, s>>>(partial, block_prefix, cams, 1.0, loss);
  return launched();
}

cudaError_t launch_masked_l1(const float* rgb, const float* target, const uint8_t* mask, const DevCam* cams,
                             int n_views, const int* block_prefix, int n_blocks, float weight, double* partial,
                             double* loss, float* d_rgb, cudaStream_t s) {
  if (n_blocks > 0) {
    l1_partial_kernel<<<n_blocks, kLossThreads, 0, s>>>(rgb, target, mask, cams, n_views, block_prefix, weight,
                                                        partial, d_rgb);
    cudaError_t e = launched();
    if (e != cudaSuccess) return e;
  }
  // the final pass divides by h*w; the L1 mean is over 3*h*w values
  bg_loss_final_kernel<<<n_views, kViewSumThreads, 0, s>>>(partial, block_prefix, cams, 1.0 / 3.0, loss);
  return launched();
}

size_t prune_words(uint32_t n) {
  const size_t tiles = ((size_t)n + kPruneThreads - 1) / kPruneThreads;
  return 2 * (tiles + (tiles + kPruneWarps - 1) / kPruneWarps);
}

cudaError_t launch_prune(const float* score, uint32_t n, float threshold, const GaussPtrs& in, int sh_degree,
                         GaussOut out, int64_t* border_idx, int64_t border_cap, uint32_t* words, uint32_t* done,
                         uint32_t* n_out, cudaStream_t s) {
  if (n == 0) return cudaMemsetAsync(n_out, 0, 2 * sizeof(uint32_t), s);
  const uint32_t tiles = (uint32_t)(((uint64_t)n + kPruneThreads - 1) / kPruneThreads);
  uint32_t* blocks = words + 2 * (size_t)tiles;
  prune_count_kernel<<<(tiles + kPruneWarps - 1) / kPruneWarps, kPruneThreads, 0, s>>>(score, n, threshold, tiles,
                                                                                      words, blocks, done, n_out);
  const cudaError_t e = launched();
  if (e != cudaSuccess) return e;
#define OCGS_PRUNE(D) \
  prune_copy_kernel<D><<<tiles, kPruneThreads, 0, s>>>(score, n, threshold, in, out, border_idx, border_cap, \
                                                       reinterpret_cast<const uint2*>(words),                \
                                                       reinterpret_cast<const uint2*>(blocks))
  switch (sh_degree) {
    case 0: OCGS_PRUNE(0); break;
    case 1: OCGS_PRUNE(1); break;
    case 2: OCGS_PRUNE(2); break;
    default: OCGS_PRUNE(3); break;
  }
#undef OCGS_PRUNE
  return launched();
}

}  // namespace ocgs

// ----------------------------------------------------------------------------- allocation-free background loss
//
// ocgs_background_loss_noalloc computes exactly what ocgs_background_loss
// computes, with the same kernels, but needs no context and allocates no
// device memory: its scratch (the per-block FP64 partial sums, the view table
// and the block prefix) lives in one file-scope device array of fixed size,
// which every GPU that loads this library holds until the process exits.
// Host code cannot hand that array to a kernel by name (in host code the name
// is only a stand-in), so the first call on each device, with that device
// current, looks its device address up with cudaGetSymbolAddress and keeps it.
// The view sizes travel to the device as a kernel argument (copied by value
// at launch), and a one-block kernel writes the view table and the block
// prefix into the array, so no host buffer is read after the call returns.
namespace {

constexpr int kNoAllocMaxViews = 1024;
constexpr int kNoAllocMaxBlocks = 65536;  // 65536 blocks x 4096 pixels = 268,435,456 pixels per call
constexpr size_t kNoAllocPartialBytes = sizeof(double) * kNoAllocMaxBlocks;
constexpr size_t kNoAllocCamOffset = kNoAllocPartialBytes;
constexpr size_t kNoAllocCamBytes = ((sizeof(ocgs::DevCam) * kNoAllocMaxViews) + 255) & ~(size_t)255;
constexpr size_t kNoAllocPrefixOffset = kNoAllocCamOffset + kNoAllocCamBytes;
constexpr size_t kNoAllocBytes = kNoAllocPrefixOffset + sizeof(int) * (kNoAllocMaxViews + 1);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// width and height of every view (each at most 16384), passed by value
struct NoAllocViews {
  uint16_t w[kNoAllocMaxViews];
  uint16_t h[kNoAllocMaxViews];
};

// One block of kNoAllocMaxViews threads: thread v fills the view table entry of
// view v (size and first pixel) and the block prefix (first loss block of v).
__global__ void __launch_bounds__(kNoAllocMaxViews) noalloc_setup_kernel(const NoAllocViews views, int n_views,
                                                                         ocgs::DevCam* __restrict__ cams,
                                                                         int* __restrict__ prefix) {
  __shared__ long long s_pix[kNoAllocMaxViews];
  __shared__ int s_blk[kNoAllocMaxViews];
  const int v = threadIdx.x;
  const long long np = v < n_views ? (long long)views.w[v] * views.h[v] : 0;
  s_pix[v] = np;
  s_blk[v] = (int)((np + ocgs::kLossBlockPixels - 1) / ocgs::kLossBlockPixels);
  __syncthreads();
  // inclusive Hillis-Steele scan over the views
  for (int o = 1; o < kNoAllocMaxViews; o <<= 1) {
    const long long pp = v >= o ? s_pix[v - o] : 0;
    const int bb = v >= o ? s_blk[v - o] : 0;
    __syncthreads();
    s_pix[v] += pp;
    s_blk[v] += bb;
    __syncthreads();
  }
  if (v < n_views) {
    ocgs::DevCam d;
    memset(&d, 0, sizeof(d));
    d.W = views.w[v];
    d.H = views.h[v];
    d.pix_offset = s_pix[v] - np;
    cams[v] = d;
    prefix[v] = s_blk[v] - (int)((np + ocgs::kLossBlockPixels - 1) / ocgs::kLossBlockPixels);
  }
  if (v == n_views - 1) prefix[n_views] = s_blk[v];
}

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_addr[kNoAllocMaxDevices];  // device address of the array, per device

}  // namespace

extern "C" ocgs_status ocgs_background_loss_noalloc(const float* alpha, const uint8_t* mask,
                                                    const ocgs_camera* cams, int32_t n_views, float gamma,
                                                    double* loss, float* d_alpha, void* stream) {
  if (!alpha || !mask || !loss || !cams) return OCGS_ERR_ARG;
  if (n_views < 1) return OCGS_ERR_ARG;
  if (n_views > kNoAllocMaxViews) return OCGS_ERR_CAPACITY;  // beyond the static view table
  if (!std::isfinite(gamma)) return OCGS_ERR_ARG;
  NoAllocViews views;
  int64_t blocks = 0;
  for (int v = 0; v < n_views; ++v) {
    if (cams[v].width < 1 || cams[v].height < 1 || cams[v].width > 16384 || cams[v].height > 16384)
      return OCGS_ERR_ARG;
    const int64_t np = (int64_t)cams[v].width * cams[v].height;
    blocks += (np + ocgs::kLossBlockPixels - 1) / ocgs::kLossBlockPixels;
    views.w[v] = (uint16_t)cams[v].width;
    views.h[v] = (uint16_t)cams[v].height;
  }
  if (blocks > kNoAllocMaxBlocks) return OCGS_ERR_CAPACITY;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return OCGS_ERR_CUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return OCGS_ERR_ARG;
  const cudaStream_t s = static_cast<cudaStream_t>(stream);
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mutex);
    if (!g_noalloc_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return OCGS_ERR_CUDA;
      g_noalloc_addr[dev] = static_cast<unsigned char*>(p);
    }
    base = g_noalloc_addr[dev];
  }
  ocgs::DevCam* d_cams = reinterpret_cast<ocgs::DevCam*>(base + kNoAllocCamOffset);
  int* d_prefix = reinterpret_cast<int*>(base + kNoAllocPrefixOffset);
  double* d_partial = reinterpret_cast<double*>(base);
  noalloc_setup_kernel<<<1, kNoAllocMaxViews, 0, s>>>(views, n_views, d_cams, d_prefix);
  if (ocgs::launched() != cudaSuccess) return OCGS_ERR_CUDA;
  if (ocgs::launch_background_loss(alpha, mask, d_cams, n_views, d_prefix, (int)blocks, gamma, d_partial, loss,
                                   d_alpha, s) != cudaSuccess)
    return OCGS_ERR_CUDA;
  return OCGS_OK;
}
