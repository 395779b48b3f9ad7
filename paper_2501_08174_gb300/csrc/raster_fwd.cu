// Forward tile rasterizer: front-to-back compositing (Sec. 4.3) with the
// optional per-Gaussian contribution record (Sec. 4.3, Sec. 5.1).
//
// A warp owns one band of a screen tile (32 threads x PPT vertically adjacent
// pixels each: full tile rows) and walks the tile's sorted (depth, Gaussian)
// list on its own, with no CTA barrier: its own slot of the persistent queue,
// its own shared-memory batches of BATCH records.  Every lane evaluates the
// batch against its pixel centres, so one shared-memory read of a record
// serves PPT pixels; the batch staging first drops, in order, the entries
// whose support misses the band's rows.  Compositing of a pixel stops at the
// first blended candidate that would bring its transmittance below 1e-4
// (rendering ends once the pixel reaches an opacity close to 1), and a warp
// stops once all its pixels have stopped.  The forward optionally records, for
// each Gaussian, the max blending weight over the pixels where it was blended
// (the per-Gaussian visibility record kept while colours accumulate), with
// one warp max-reduction per entry and one flush per batch.
#include "raster_common.cuh"

namespace ocgs {
namespace {
using namespace raster;

#ifdef OCGS_COUNT
__device__ unsigned long long g_diag[2];  // warp-entries, (pixel, entry) blends
#endif

// Resident warps per SM the compiler is asked to fit (caps registers per
// thread): 20 leaves 96 registers, enough for the image planes without spills
// (24 warps at 80 registers spill about 60 bytes and measured 1.5 % slower).
#ifndef OCGS_FWD_WARPS
#define OCGS_FWD_WARPS 20
#endif
// With the Q plane 20 would spill; 16 measured 3 % faster (28.7 -> 27.5 ms on 1M surfels x 64 views).
#ifndef OCGS_FWD_WARPS_Q2
#define OCGS_FWD_WARPS_Q2 16
#endif
// A pass without images holds half the registers (1.89 -> 1.86 ms on 500k Gaussians x 16 views).
#ifndef OCGS_SWEEP_WARPS
#define OCGS_SWEEP_WARPS 28
#endif

// Q2: also accumulate Q = sum w z^2 (the depth distortion's third plane)
// EWA: the records are projected 3D Gaussians (the 3DGS variant of Appendix B)
template <int TW, int TH, int PPT, int BATCH, bool IMG, bool SCORE, bool Q2, bool EWA>
__global__ void __launch_bounds__(kBlockWarps * 32, (!IMG ? OCGS_SWEEP_WARPS : Q2 ? OCGS_FWD_WARPS_Q2 : OCGS_FWD_WARPS) / kBlockWarps)
    raster_fwd_kernel(const RasterArgs a) {
  constexpr int WPT = TW * TH / PPT / 32;  // warps per tile: each owns a band of full tile rows
  using B = Batch<BATCH>;
  constexpr bool kPrefetch = IMG && B::kRounds == 1;
  // The exact band test in the staging: worth its registers where no images are held (sweep of
  // 300k surfels x 100 views 14.3 -> 13.1 ms; with images it spills, 2.72 -> 2.83 ms) and the
  // support is not the near-disc of a projected 3D Gaussian (1.85 -> 2.00 ms).
  constexpr bool kBandTest = !IMG && !EWA;
  __shared__ float4 s_g0[kBlockWarps][BATCH], s_g1[kBlockWarps][BATCH], s_g2[kBlockWarps][BATCH],
      s_a0[kBlockWarps][IMG ? BATCH : 1];
  // (n_y, n_z, blend bound, list position + 1); a pass without images keeps the bound in g0.w
  __shared__ float4 s_b[kBlockWarps][IMG ? BATCH : 1];
  __shared__ uint32_t s_gid[kBlockWarps][SCORE ? BATCH : 1];
  __shared__ unsigned s_max[kBlockWarps][SCORE ? BATCH : 1];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const uint32_t n_units = (a.n_queue ? *a.n_queue : a.n_tiles) * (uint32_t)WPT;
  for (uint32_t it = 0;; ++it) {
    // work unit: one warp's band of one tile; the warps run independently
    uint32_t unit;
    if (a.persistent_ctas) {
      uint32_t u = 0;
      if (lane == 0) u = atomicAdd(a.queue, 1u);
      unit = __shfl_sync(kFull, u, 0);
      if (unit >= n_units) break;
    } else {
      if (it > 0) break;
      unit = blockIdx.x * kBlockWarps + wib;
      if (unit >= n_units) break;
    }
    uint32_t tile = unit / WPT;
    if (a.persistent_ctas && a.tile_order) tile = a.tile_order[tile];
    const int tid = (int)(unit % WPT) * 32 + lane;  // thread of the tile
    const int lx = tid % TW, ly0 = (tid / TW) * PPT;  // this thread's column and first of PPT rows
    const int v = view_of_tile(a.tile_prefix, a.n_views, (int)tile);
    const DevCam& cam = a.cams[v];
    const int local = (int)tile - cam.tile_offset;
    const int px = (local % cam.tiles_x) * TW + lx;
    const int py0 = (local / cam.tiles_x) * TH + ly0;
    const float pxf = (float)px + 0.5f;
    const uint2 rg = a.ranges[tile];
    const uint32_t start = rg.x, end = rg.y;
    const int64_t gbase = (int64_t)v * a.n_gauss;
    // pixel k of this thread is lane (k & 1) of pair k / 2; an odd PPT leaves a
    // dummy lane that starts done
    constexpr int NP = (PPT + 1) / 2;
    float2 T[NP], c0[NP], c1[NP], c2[NP], dep[NP], n0[NP], n1[NP], n2[NP], qz[NP];
    uint32_t last[2 * NP];
    bool done[2 * NP];
    bool alldone = true;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T[p] = bc2(1.f);
      c0[p] = c1[p] = c2[p] = dep[p] = n0[p] = n1[p] = n2[p] = qz[p] = bc2(0.f);
    }
#pragma unroll
    for (int k = 0; k < 2 * NP; ++k) {
      last[k] = 0u;
      done[k] = !(k < PPT && px < cam.W && py0 + k < cam.H);
    }
    uint32_t pos0 = 0u;  // list position before this pass's first entry
    if (a.prior) {
      // second pass: continue each pixel from the end of the tile's first-pass list
      const uint2 pr = a.prior[tile];
      pos0 = pr.y - pr.x;
#pragma unroll
      for (int k = 0; k < PPT; ++k) {
        if (!done[k]) {
          const int64_t pix = cam.pix_offset + (int64_t)(py0 + k) * cam.W + px;
          const int p = k >> 1, i = k & 1;
          set_lane2(T[p], i, a.t_final[pix]);
          if (IMG) {
            set_lane2(c0[p], i, a.out.rgb[3 * pix]);
            set_lane2(c1[p], i, a.out.rgb[3 * pix + 1]);
            set_lane2(c2[p], i, a.out.rgb[3 * pix + 2]);
            set_lane2(dep[p], i, a.out.depth[pix]);
            if (Q2) set_lane2(qz[p], i, a.out.depth2[pix]);
            set_lane2(n0[p], i, a.out.normal[3 * pix]);
            set_lane2(n1[p], i, a.out.normal[3 * pix + 1]);
            set_lane2(n2[p], i, a.out.normal[3 * pix + 2]);
          }
          if (a.last) last[k] = a.last[pix];
          done[k] = a.done[pix] != 0;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2 * NP; ++k) alldone = alldone && done[k];
    const float4 band = warp_band<TW, TH, PPT>(cam, local, (int)(unit % WPT));
    const float2 pyb = make_float2((float)py0 + 0.5f, (float)py0 + 1.5f);
    // the next batch's list entries are requested while the current one is processed
    uint32_t nidx = 0;
    if (kPrefetch && lane < B::kLanes && start + lane < end) nidx = a.vals[start + lane];
    for (uint32_t b0 = start; b0 < end; b0 += BATCH) {
      if (__all_sync(kFull, alldone)) break;
      __syncwarp();  // the previous batch is consumed
      // a batch of the list; keep (in order) the entries whose rows meet this warp's band
      int cnt = 0;
#pragma unroll
      for (int r = 0; r < B::kRounds; ++r) {
        const uint32_t kk = b0 + (uint32_t)(r * 32 + lane);
        bool keep = false;
        uint32_t idx = 0;
        float4 a1 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < B::kLanes && kk < end) {
          idx = kPrefetch ? nidx : a.vals[kk];
          a1 = a.rec.a1[idx];
          keep = a1.w >= band.z && a1.z <= band.w;
        }
        float4 g0, g1, g2;
        if (kBandTest && keep) {
          g0 = a.rec.g0[idx];
          g1 = a.rec.g1[idx];
          g2 = a.rec.g2[idx];
          keep = meets_band(g0, g1, g2, band, cam);
        }
        const unsigned km = __ballot_sync(kFull, keep);
        if (keep) {
          const int slot = cnt + __popc(km & lt);
          if (!kBandTest) {
            g0 = a.rec.g0[idx];
            g1 = a.rec.g1[idx];
            g2 = a.rec.g2[idx];
          }
          if (!IMG) g0.w = blend_rho(g0.z);  // the centre depth is not needed: the blend bound takes its place
          s_g0[wib][slot] = g0;
          s_g1[wib][slot] = g1;
          s_g2[wib][slot] = g2;
          if (IMG) {
            s_a0[wib][slot] = a.rec.a0[idx];
            s_b[wib][slot] = make_float4(a1.x, a1.y, blend_rho(g0.z), __uint_as_float(pos0 + kk - start + 1u));
          }
          if (SCORE) s_gid[wib][slot] = (uint32_t)((int64_t)idx - gbase);
        }
        cnt += __popc(km);
      }
      if (kPrefetch && lane < B::kLanes && b0 + BATCH + lane < end) nidx = a.vals[b0 + BATCH + lane];
      __syncwarp();
      int j = 0;
      for (; j < cnt; ++j) {
        if ((j & 7) == 0 && j > 0 && __all_sync(kFull, alldone)) break;
        const float4 g0 = s_g0[wib][j], g1 = s_g1[wib][j], g2 = s_g2[wib][j];
        const SplatColumn col = splat_column(g0, g1, g2, pxf);
        float4 ap = make_float4(0.f, 0.f, 0.f, 0.f), an = ap;
        if (IMG) {
          ap = s_a0[wib][j];
          an = s_b[wib][j];
        }
        const float rb = IMG ? an.z : g0.w;
        const uint32_t pos = __float_as_uint(an.w);
        // Every lane evaluates every pair, without a branch per pair or per lane: a candidate
        // that is not blended, or whose pixel has stopped, has alpha = 0 (T (1 - 0) = T, w = 0
        // exactly).  All pairs are evaluated before one test asks whether any of their pixels
        // stops here, and only then summed: the pairs' dependency chains interleave, and the
        // rare stop costs one branch per entry (500k surfels x 16 views: 3.35 -> 2.78 ms with
        // the batch-wide score flush, against a branch per lane and a stop test per pair).
        float2 Tn[NP], w[NP], z[NP];
        bool ok[2 * NP];
        float tmin = 1.f;
#ifdef OCGS_COUNT
        if (lane == 0) OCGS_DIAG(0, 1);
#endif
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const int k0 = 2 * p, k1 = 2 * p + 1;
          const float2 py = padd(pyb, bc2((float)(2 * p)));  // exact: half-integers below 2^15
          const SplatHead2 h = splat_head2(g0, g1, g2, col, py);
          const SplatEval2 e = splat_tail2<false, EWA>(g0, g2, h, rb, !done[k0], !done[k1]);
          Tn[p] = pmul(T[p], pfma(e.alpha, bc2(-1.f), bc2(1.f)));  // T (1 - alpha)
          w[p] = pmul(e.alpha, T[p]);
          z[p] = e.z;
          ok[k0] = e.ok[0];
          ok[k1] = e.ok[1];
          tmin = fminf(tmin, fminf(Tn[p].x, Tn[p].y));
        }
        if (tmin < kTEps) {
          // an entry that would take T below kTEps ends the pixel unblended
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            if (Tn[p].x < kTEps) { done[2 * p] = true; w[p].x = 0.f; Tn[p].x = T[p].x; ok[2 * p] = false; }
            if (Tn[p].y < kTEps) { done[2 * p + 1] = true; w[p].y = 0.f; Tn[p].y = T[p].y; ok[2 * p + 1] = false; }
          }
          alldone = true;
#pragma unroll
          for (int k = 0; k < 2 * NP; ++k) alldone = alldone && done[k];
        }
        float wmax = 0.f;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          if (ok[2 * p]) last[2 * p] = pos;
          if (ok[2 * p + 1]) last[2 * p + 1] = pos;
          if (IMG) {
            c0[p] = pfma(w[p], bc2(ap.x), c0[p]);
            c1[p] = pfma(w[p], bc2(ap.y), c1[p]);
            c2[p] = pfma(w[p], bc2(ap.z), c2[p]);
            dep[p] = pfma(w[p], z[p], dep[p]);
            if (Q2) qz[p] = pfma(pmul(w[p], z[p]), z[p], qz[p]);
            n0[p] = pfma(w[p], bc2(ap.w), n0[p]);
            n1[p] = pfma(w[p], bc2(an.x), n1[p]);
            n2[p] = pfma(w[p], bc2(an.y), n2[p]);
          }
          T[p] = Tn[p];
          if (SCORE) wmax = fmaxf(wmax, fmaxf(w[p].x, w[p].y));
#ifdef OCGS_COUNT
          OCGS_DIAG(1, (w[p].x > 0.f ? 1 : 0) + (w[p].y > 0.f ? 1 : 0));
#endif
        }
        if (SCORE) {
          // the warp's largest weight of the entry (non-negative floats order like their bits)
          const unsigned m = __reduce_max_sync(kFull, __float_as_uint(wmax));
          if (lane == 0) s_max[wib][j] = m;
        }
      }
      if (SCORE) {
        // the batch's maxima, one entry per lane: at most one atomic per entry and warp
        __syncwarp();
#pragma unroll
        for (int r = 0; r < B::kRounds; ++r) {
          const int e = r * 32 + lane;
          if (e < j) {
            const unsigned m = s_max[wib][e];
            if (m) atomicMax(reinterpret_cast<unsigned*>(a.score) + s_gid[wib][e], m);
          }
        }
      }
    }
    if (a.open) {
      // the tile stays open if a pixel of any of its warps has not stopped within its list
      if (__any_sync(kFull, !alldone) && lane == 0) a.open[tile] = 1u;
      if (!IMG) {
        // a pass without images keeps only what the continuation needs: T and the stop flags
#pragma unroll
        for (int k = 0; k < PPT; ++k) {
          if (px < cam.W && py0 + k < cam.H) {
            const int64_t pix = cam.pix_offset + (int64_t)(py0 + k) * cam.W + px;
            a.t_final[pix] = lane2(T[k >> 1], k & 1);
            a.done[pix] = done[k] ? 1 : 0;
          }
        }
      }
    }
    if (IMG) {
#pragma unroll
      for (int k = 0; k < PPT; ++k) {
        const int py = py0 + k;
        const int p = k >> 1, i = k & 1;
        if (px < cam.W && py < cam.H) {
          const int64_t pix = cam.pix_offset + (int64_t)py * cam.W + px;
          const float Tk = lane2(T[p], i);
          a.out.rgb[3 * pix + 0] = lane2(c0[p], i);
          a.out.rgb[3 * pix + 1] = lane2(c1[p], i);
          a.out.rgb[3 * pix + 2] = lane2(c2[p], i);
          a.out.alpha[pix] = 1.f - Tk;
          a.out.depth[pix] = lane2(dep[p], i);
          if (Q2) a.out.depth2[pix] = lane2(qz[p], i);
          a.out.normal[3 * pix + 0] = lane2(n0[p], i);
          a.out.normal[3 * pix + 1] = lane2(n1[p], i);
          a.out.normal[3 * pix + 2] = lane2(n2[p], i);
          // the state of the backward, or (T alone) of a second pass, when the pass keeps it
          if (a.t_final) a.t_final[pix] = Tk;
          if (a.last) a.last[pix] = last[k];
          if (a.open) a.done[pix] = done[k] ? 1 : 0;
        }
      }
    }
  }
}

template <int TW, int TH, int PPT, int BATCH>
cudaError_t fwd_dispatch(const RasterArgs& a, bool img, cudaStream_t s) {
  const unsigned grid = warp_grid<TW, TH, PPT>(a.persistent_ctas, a.n_tiles);
  if (grid == 0) return cudaSuccess;
  constexpr int NT = kBlockWarps * 32;
  const bool score = a.score != nullptr;
  const bool q2 = img && a.out.depth2 != nullptr;
  if (a.ewa) {
    if (img && score) raster_fwd_kernel<TW, TH, PPT, BATCH, true, true, false, true><<<grid, NT, 0, s>>>(a);
    else if (img) raster_fwd_kernel<TW, TH, PPT, BATCH, true, false, false, true><<<grid, NT, 0, s>>>(a);
    else if (score) raster_fwd_kernel<TW, TH, PPT, BATCH, false, true, false, true><<<grid, NT, 0, s>>>(a);
    else return cudaSuccess;
  } else if (img && score && q2) raster_fwd_kernel<TW, TH, PPT, BATCH, true, true, true, false><<<grid, NT, 0, s>>>(a);
  else if (img && q2) raster_fwd_kernel<TW, TH, PPT, BATCH, true, false, true, false><<<grid, NT, 0, s>>>(a);
  else if (img && score) raster_fwd_kernel<TW, TH, PPT, BATCH, true, true, false, false><<<grid, NT, 0, s>>>(a);
  else if (img) raster_fwd_kernel<TW, TH, PPT, BATCH, true, false, false, false><<<grid, NT, 0, s>>>(a);
  else if (score) raster_fwd_kernel<TW, TH, PPT, BATCH, false, true, false, false><<<grid, NT, 0, s>>>(a);
  else return cudaSuccess;
  return launched();
}

__global__ void sum_u32_kernel(const uint32_t* __restrict__ v, int64_t n, unsigned long long* __restrict__ out) {
  unsigned long long acc = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += v[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

}  // namespace

#ifdef OCGS_COUNT
extern "C" int ocgs_diag_read(unsigned long long* out, int reset) {
  cudaMemcpyFromSymbol(out, g_diag, sizeof(g_diag));
  if (reset) {
    unsigned long long z[2] = {0};
    cudaMemcpyToSymbol(g_diag, z, sizeof(z));
  }
  return 0;
}
#endif

cudaError_t launch_sum_u32(const uint32_t* v, int64_t n, unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
  if (e != cudaSuccess || n == 0) return e;
  sum_u32_kernel<<<304, 256, 0, s>>>(v, n, out);
  return launched();
}

cudaError_t launch_raster_forward(const RasterArgs& a, int tile_w, int tile_h, int ppt, int batch, bool write_image,
                                  cudaStream_t s) {
#define OCGS_FWD(W, H, K, BT) \
  if (tile_w == W && tile_h == H && ppt == K && batch == BT) return fwd_dispatch<W, H, K, BT>(a, write_image, s);
  OCGS_RASTER_SHAPES(OCGS_FWD)
#undef OCGS_FWD
  return cudaErrorInvalidValue;
}

}  // namespace ocgs
