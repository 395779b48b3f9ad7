// Backward tile rasterizer: the reverse-order adjoint of the front-to-back
// compositing (the backpropagation through the rasterizer of Sec. 3.2).
//
// The backward walks each tile's list back to front from each pixel's last
// blended entry, recovering the transmittance T_i = T_{i+1} / (1 - alpha_i)
// from the stored final transmittance, so nothing per (pixel, Gaussian) is
// stored between the passes.  Per-Gaussian gradients are summed over the
// thread's pixels, reduced over the warp, gathered per batch in the warp's
// shared memory and added to global memory with one vector atomic per 4
// values, entry and warp.  The warp reduction goes through shared memory (see
// warp_totals).
//
// Terms that are linear in per-entry or per-column constants are summed before
// they are multiplied: a thread sums the pixel terms of its column and scales
// the sums by the column offset dx once per entry, and the centre gradient's
// share through (u, v, den) is formed from the warp totals of the u, v and den
// terms when the batch is flushed.
#include "raster_common.cuh"

namespace ocgs {
namespace {
using namespace raster;

#ifdef OCGS_COUNT
__device__ unsigned long long g_diag[2];  // warp-entries, (pixel, entry) blends
#endif

// Resident warps per SM the compiler is asked to fit (caps registers per thread): 20 leaves
// 96 registers; 16 measured 0.4 % and 24 (spills) 5 % slower on 500k surfels x 16 views
#ifndef OCGS_BWD_WARPS
#define OCGS_BWD_WARPS 20
#endif
// With depth and normal cotangents: 16 resident warps leave 128 registers; 20 spill (62.8
// against 54.9 ms on 1M surfels x 64 views)
#ifndef OCGS_BWD_WARPS_GEO
#define OCGS_BWD_WARPS_GEO 16
#endif
// warps per CTA of the backward (the resident-warp targets are multiples of it)
#ifndef OCGS_BWD_BLOCK_WARPS
#define OCGS_BWD_BLOCK_WARPS 4
#endif
constexpr int kBW = OCGS_BWD_BLOCK_WARPS;
static_assert(OCGS_BWD_WARPS % kBW == 0 && OCGS_BWD_WARPS_GEO % kBW == 0, "resident warps per CTA");

// Two sums beside the gradient slots, kept in the row's padding until the
// flush: the totals of the u and v terms, 2 dL/drho (u, v) / den^2, from
// which the flush forms the centre gradient's share through (u, v, den).
constexpr int kSumU = 18, kSumV = 19;
static_assert(kSumV < kGradStride && kGradSlots <= kSumU, "sums in the row padding");

// Sums of the 15-sum path in the order of the reduction buffer: the 13 slots,
// then the u and v totals.
constexpr int kRedSums = kGradSlotsRGB + 2;
__device__ __forceinline__ int red_target(int q) { return q < kGradSlotsRGB ? q : kSumU + (q - kGradSlotsRGB); }

// Reduction buffer of a warp: for each of S sums two rows (the values of lanes
// 0-15 and of lanes 16-31), each 16 floats at a stride of 20.  The upper rows
// start 16 banks after the lower ones (modulo 32), so a store of one sum by all
// lanes hits every bank once, and the 16-byte loads, eight consecutive rows per
// phase, are free of conflicts.
//
// What bounds it: shared-memory wavefronts.  The 15 sums of the two pixel lanes
// stored as pairs and read back with 16 64-bit loads took 62 wavefronts per entry
// (about 3 ms of a 5.1 ms launch at one wavefront per cycle and SM on 500k
// surfels x 16 views); added first and read back with four 16-byte loads they
// take 31, and the launch 4.34 ms against 4.68.  The 20 sums of the depth and
// normal form took a transpose of 41 shuffles before (64.3 -> 63.3 ms on 1M
// surfels x 64 views).
constexpr int kRedStride = 20;
constexpr int red_upper(int s) { return s * kRedStride + (48 - s * kRedStride % 32) % 32; }
// one row more than the sums have: the lanes without a sum read past the upper rows
constexpr int red_floats(int s) { return red_upper(s) + (s + 1) * kRedStride; }

// Stores the S per-lane sums v(q) and returns, in lane L and in lane L ^ 16, the
// warp total of sum L & 15 (lane 15: undefined for S = 15).  Ends before the
// reads of other lanes are ordered: the caller synchronises before the next call.
template <int S, class F>
__device__ __forceinline__ float warp_totals(float* red, int lane, F v) {
  float* wr = red + (lane >> 4) * red_upper(S) + (lane & 15);
#pragma unroll
  for (int q = 0; q < S; ++q) wr[q * kRedStride] = v(q);
  __syncwarp();
  const float4* rd = reinterpret_cast<const float4*>(red + (lane >> 4) * red_upper(S) + (lane & 15) * kRedStride);
  float4 t = rd[0];
#pragma unroll
  for (int i = 1; i < 4; ++i) {
    const float4 b = rd[i];
    const float2 lo = padd(make_float2(t.x, t.y), make_float2(b.x, b.y));
    const float2 hi = padd(make_float2(t.z, t.w), make_float2(b.z, b.w));
    t = make_float4(lo.x, lo.y, hi.x, hi.y);
  }
  const float2 u = padd(make_float2(t.x, t.y), make_float2(t.z, t.w));
  const float tot = __fadd_rn(u.x, u.y);
  return __fadd_rn(tot, __shfl_xor_sync(kFull, tot, 16));
}

// Slots accumulated with the opposite sign (flipped when the lanes are summed).
__device__ __forceinline__ bool negated_slot(int q) { return q == kGe0 || q == kGe1 || q == kGe2; }

// GEO: a depth, depth2 or normal cotangent is given; without one the depth and
// normal terms of the adjoint are zero and are not evaluated (13 slots instead
// of 18, 15 sums instead of 20).
template <int TW, int TH, int PPT, int BATCH, bool GEO>
__global__ void __launch_bounds__(kBW * 32, (GEO ? OCGS_BWD_WARPS_GEO : OCGS_BWD_WARPS) / kBW)
    raster_bwd_kernel(const RasterBwdArgs a) {
  constexpr int WPT = TW * TH / PPT / 32;  // warps per tile: each owns a band of full tile rows
  constexpr int ROWS = BATCH > 32 ? BATCH / 32 : 1;  // gradient rows of a batch each lane flushes
  using B = Batch<BATCH>;
  __shared__ float4 s_g0[kBW][BATCH], s_g1[kBW][BATCH], s_g2[kBW][BATCH], s_a0[kBW][BATCH];
  // (n_y, n_z, blend bound, list position); the colour and opacity form, which needs neither
  // normals nor depths, keeps the last two in the depth fields of g0 and g2
  __shared__ float4 s_b[kBW][GEO ? BATCH : 1];
  __shared__ uint32_t s_idx[kBW][BATCH];
  __shared__ __align__(16) float s_grad[kBW][BATCH * kGradStride];  // per-batch gradient sums of each entry
  __shared__ __align__(16) float s_red[kBW][red_floats(GEO ? kGradStride : kRedSums)];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    if (r * 32 + lane < BATCH) {  // a batch of 16 has rows for half the lanes
      float* row = &s_grad[wib][(r * 32 + lane) * kGradStride];
#pragma unroll
      for (int q = 0; q < kGradStride; ++q) row[q] = 0.f;
    }
  }
  // the sign of the sum this lane holds after the reduction, and (15-sum form) its place in the row
  const float red_sign = negated_slot(lane & 15) ? -1.f : 1.f;
  const int red_dst = red_target(lane & 15);
  const uint32_t n_units = a.n_tiles * (uint32_t)WPT;
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
      unit = blockIdx.x * kBW + wib;
      if (unit >= n_units) break;
    }
    uint32_t tile = unit / WPT;
    if (a.persistent_ctas && a.tile_order) tile = a.tile_order[tile];
    const int tid = (int)(unit % WPT) * 32 + lane;  // thread of the tile
    const int lx = tid % TW, ly0 = (tid / TW) * PPT;
    const int v = view_of_tile(a.tile_prefix, a.n_views, (int)tile);
    const DevCam& cam = a.cams[v];
    const int local = (int)tile - cam.tile_offset;
    const int px = (local % cam.tiles_x) * TW + lx;
    const int py0 = (local / cam.tiles_x) * TH + ly0;
    const float pxf = (float)px + 0.5f;
    const uint2 rg1 = a.ranges[tile];
    const uint32_t start = rg1.x;
    // a two-pass list continues in the second segment after its first rg1.y - rg1.x entries
    const uint32_t len1 = a.ranges2 ? rg1.y - rg1.x : 0xffffffffu;
    const uint32_t start2 = a.ranges2 ? a.ranges2[tile].x : 0u;
    // pixel k of this thread is lane (k & 1) of pair k / 2 (an odd PPT leaves an idle lane)
    constexpr int NP = (PPT + 1) / 2;
    float2 T[NP], gAT[NP], S[NP];
    float2 gC0[NP], gC1[NP], gC2[NP], gD[NP], gN0[NP], gN1[NP], gN2[NP], gQ[NP];
    uint32_t last[2 * NP];
    uint32_t thread_last = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      T[p] = bc2(1.f);
      gAT[p] = bc2(0.f);
      S[p] = bc2(0.f);  // sum over later blended entries of w * (gC.rgb + gD z + gN.n)
      gC0[p] = gC1[p] = gC2[p] = gD[p] = gN0[p] = gN1[p] = gN2[p] = gQ[p] = bc2(0.f);
    }
#pragma unroll
    for (int k = 0; k < 2 * NP; ++k) {
      last[k] = 0u;
      const int py = py0 + k;
      const int p = k >> 1, i = k & 1;
      if (k < PPT && px < cam.W && py < cam.H) {
        const int64_t pix = cam.pix_offset + (int64_t)py * cam.W + px;
        const float Tf = a.t_final[pix];
        set_lane2(T[p], i, Tf);
        last[k] = a.last[pix];
        if (a.d_out.rgb) {
          set_lane2(gC0[p], i, a.d_out.rgb[3 * pix]);
          set_lane2(gC1[p], i, a.d_out.rgb[3 * pix + 1]);
          set_lane2(gC2[p], i, a.d_out.rgb[3 * pix + 2]);
        }
        if (a.d_out.alpha) set_lane2(gAT[p], i, a.d_out.alpha[pix] * Tf);
        if (GEO && a.d_out.depth) set_lane2(gD[p], i, a.d_out.depth[pix]);
        if (GEO && a.d_out.depth2) set_lane2(gQ[p], i, a.d_out.depth2[pix]);
        if (GEO && a.d_out.normal) {
          set_lane2(gN0[p], i, a.d_out.normal[3 * pix]);
          set_lane2(gN1[p], i, a.d_out.normal[3 * pix + 1]);
          set_lane2(gN2[p], i, a.d_out.normal[3 * pix + 2]);
        }
        thread_last = max(thread_last, last[k]);
      }
    }
    // entries at or beyond the warp's largest last index are idle for every lane
    const int warp_last = (int)__reduce_max_sync(kFull, thread_last);
    const float4 band = warp_band<TW, TH, PPT>(cam, local, (int)(unit % WPT));
    auto list_at = [&](int q) { return (uint32_t)q < len1 ? a.vals[start + q] : a.vals2[start2 + ((uint32_t)q - len1)]; };
    const float2 pyb = make_float2((float)py0 + 0.5f, (float)py0 + 1.5f);
    // the next batch's list entries are requested while the current one is processed
    uint32_t nidx = 0;
    if (B::kRounds == 1) {
      const int q = max(0, warp_last - BATCH) + lane;
      if (lane < B::kLanes && q < warp_last) nidx = list_at(q);
    }
    for (int bend = warp_last; bend > 0; bend -= BATCH) {
      const int bstart = max(0, bend - BATCH);
      __syncwarp();  // the previous batch is consumed and flushed
      // a batch of the list, ending at bend; keep (in order) the entries whose rows meet the band
      int cnt = 0;
#pragma unroll
      for (int r = 0; r < B::kRounds; ++r) {
        const int q = bstart + r * 32 + lane;
        bool keep = false;
        uint32_t idx = 0;
        float4 a1 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < B::kLanes && q < bend) {
          idx = B::kRounds == 1 ? nidx : list_at(q);
          a1 = a.rec.a1[idx];
          keep = a1.w >= band.z && a1.z <= band.w;
        }
        float4 g0, g1, g2;
        if (keep) {
          g0 = a.rec.g0[idx];
          g1 = a.rec.g1[idx];
          g2 = a.rec.g2[idx];
          // exact band test; with one pixel per thread (few tiles) the launch waits for its longest
          // list, where the test lengthens every batch (crops: 337 -> 351 us)
          if (PPT > 1) keep = meets_band(g0, g1, g2, band, cam);
        }
        const unsigned km = __ballot_sync(kFull, keep);
        if (keep) {
          const int slot = cnt + __popc(km & lt);
          const float rb = blend_rho(g0.z);
          if (GEO) {
            s_b[wib][slot] = make_float4(a1.x, a1.y, rb, __int_as_float(q));
          } else {
            g0.w = rb;
            g2.w = __int_as_float(q);
          }
          s_g0[wib][slot] = g0;
          s_g1[wib][slot] = g1;
          s_g2[wib][slot] = g2;
          s_a0[wib][slot] = a.rec.a0[idx];
          s_idx[wib][slot] = idx;
        }
        cnt += __popc(km);
      }
      if (B::kRounds == 1) {
        const int q = max(0, bstart - BATCH) + lane;
        if (lane < B::kLanes && q < bstart) nidx = list_at(q);
      }
      __syncwarp();
      for (int j = cnt - 1; j >= 0; --j) {
#ifdef OCGS_COUNT
        if (lane == 0) OCGS_DIAG(0, 1);
#endif
        // Every entry of the walk lies before warp_last, so some lane has jj < its last index, and
        // nearly every one that passed the staging's band test blends a pixel: all are evaluated as
        // straight-line code, without a vote.  (A vote on a cheap per-pixel support test skipped one
        // entry in seven before the band test was exact; its latency and that test cost more: 4.27 ->
        // 4.16 ms on 500k surfels x 16 views, 55.6 -> 54.8 ms on 1M x 64.)
        const float4 g0 = s_g0[wib][j], g1 = s_g1[wib][j], g2 = s_g2[wib][j];
        const float4 an = GEO ? s_b[wib][j] : make_float4(0.f, 0.f, g0.w, g2.w);
        const float rb = an.z;
        const int jj = __float_as_int(an.w);  // list position
        const SplatColumn col = splat_column(g0, g1, g2, pxf);
        SplatHead2 hd[NP];
        bool live[2 * NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          const float2 py = padd(pyb, bc2((float)(2 * p)));  // exact: half-integers below 2^15
          hd[p] = splat_head2(g0, g1, g2, col, py);
          live[2 * p] = jj < (int)last[2 * p];
          live[2 * p + 1] = jj < (int)last[2 * p + 1];
        }
        const float4 ap = s_a0[wib][j];
        const float2 no = bc2(-g0.z);  // 2 dalpha/drho = -alpha = -o G
        // this thread's sums (one lane per pixel of a pair): the slots of the
        // record gradient, and the u and v totals in kSumU, kSumV.  The dx-scaled
        // slots (A00, A10, e1, and the filter term of cx) hold their pixel sums
        // until the column offset is applied after the pairs.
        // The first pair sets each sum, the others add to it.
        float2 acc[kGradStride];
        // no per-pair branch: a candidate that is not blended has alpha = 0 and
        // Gc = 0, which makes its weight and every term of its adjoint exactly 0.  (A clamp-free
        // form for records whose opacity cannot reach the clamp saved its compares and cost a
        // branch: 4.14 against 4.10 ms on 500k surfels x 16 views.)
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          auto sum_fma = [&](int q, float2 x, float2 y) { acc[q] = p == 0 ? pmul(x, y) : pfma(x, y, acc[q]); };
          auto sum_add = [&](int q, float2 x) { acc[q] = p == 0 ? x : padd(acc[q], x); };
          const SplatEval2 e = splat_tail2<true>(g0, g2, hd[p], rb, live[2 * p], live[2 * p + 1]);
#ifdef OCGS_COUNT
          OCGS_DIAG(1, (e.ok[0] ? 1 : 0) + (e.ok[1] ? 1 : 0));
#endif
          // undo the entry: T before it, its weight, and dL/dalpha
          const float2 om = pfma(e.alpha, bc2(-1.f), bc2(1.f));  // 1 - alpha
          const float2 inv = make_float2(rcp_approx(om.x), rcp_approx(om.y));
          const float2 Ti = pmul(T[p], inv);
          const float2 w = pmul(e.alpha, Ti);
          float2 F = pmul(gC0[p], bc2(ap.x));
          F = pfma(gC1[p], bc2(ap.y), F);
          F = pfma(gC2[p], bc2(ap.z), F);
          if (GEO) {
            F = pfma(gD[p], e.z, F);
            F = pfma(pmul(gQ[p], e.z), e.z, F);  // d(sum w z^2)/dw = z^2
            F = pfma(gN0[p], bc2(ap.w), F);
            F = pfma(gN1[p], bc2(an.x), F);
            F = pfma(gN2[p], bc2(an.y), F);
          }
          // dL/dalpha = T_i F + (gAT - S) / (1 - alpha)
          const float2 ga = pfma(Ti, F, pmul(pfma(S[p], bc2(-1.f), gAT[p]), inv));
          S[p] = pfma(w, F, S[p]);
          // a skipped candidate has alpha = 0, and the fast reciprocal of 1 - 0 is exactly 1
          // on this GPU (checked at 1, 2 and 0.5), so T passes through it unchanged
          T[p] = Ti;
          sum_fma(kGr, gC0[p], w);
          sum_fma(kGg, gC1[p], w);
          sum_fma(kGb, gC2[p], w);
          if (GEO) {
            sum_fma(kGnx, gN0[p], w);
            sum_fma(kGny, gN1[p], w);
            sum_fma(kGnz, gN2[p], w);
          }
          // alpha = o G below the clamp: dalpha/do = G, dalpha/drho = -o G / 2
          // (Gc is 0 at the clamp and for skipped candidates); gs2 = 2 dL/drho
          const float2 gop = pmul(ga, e.Gc);
          sum_add(kGo, gop);
          const float2 gs2 = pmul(gop, no);
          // rho and depth came from the surfel's (u, v) where it won the min, from the
          // screen-space filter elsewhere.  e.r and e.rho3 are 0 where the filter won,
          // so the surfel terms below vanish there without a mask.
          const float2 gf2 = make_float2(e.surf[0] ? 0.f : gs2.x, e.surf[1] ? 0.f : gs2.y);
          float2 gzs = bc2(0.f);
          if (GEO) {
            // d/dz of w (gD z + gQ z^2)
            const float2 gz = pmul(pfma(pmul(bc2(2.f), gQ[p]), e.z, gD[p]), w);
            gzs = make_float2(e.surf[0] ? gz.x : 0.f, e.surf[1] ? gz.y : 0.f);
            sum_add(kGzc, pfma(gzs, bc2(-1.f), gz));
            sum_fma(kGzD, gzs, e.r);
          }
          // 2 grho / den^2, shared by the u, v and den terms (rho3 = q / den^2)
          const float2 t = pmul(gs2, pmul(e.r, e.r));
          const float2 gun = pmul(t, hd[p].un);
          const float2 gvn = pmul(t, hd[p].vn);
          // -dL/dden = (2 grho rho3 + gz z) / den; the e slots accumulate negated and
          // are flipped when the lanes are summed
          const float2 ngden = GEO ? pmul(pfma(gs2, e.rho3, pmul(gzs, e.z)), e.r)
                                   : pmul(t, pmul(hd[p].q, e.r));
          sum_add(kSumU, gun);
          sum_add(kSumV, gvn);
          sum_fma(kGA01, gun, hd[p].dy);
          sum_fma(kGA11, gvn, hd[p].dy);
          sum_add(kGe0, ngden);
          sum_fma(kGe2, ngden, hd[p].dy);
          // the filter term: d rho2 / d(c) = -4 (x - c) with rho2 = 2 |x - c|^2 (the
          // factor -2 and dx are applied later)
          sum_add(kGcx, gf2);
          sum_fma(kGcy, gf2, hd[p].dy);
        }
        // the column offset of this thread's pixels
        const float2 dx = bc2(col.dx);
        acc[kGA00] = pmul(acc[kSumU], dx);
        acc[kGA10] = pmul(acc[kSumV], dx);
        acc[kGe1] = pmul(acc[kGe0], dx);
        acc[kGcx] = pmul(acc[kGcx], dx);
        float* sums = &s_grad[wib][j * kGradStride];
        auto value = [&](int q) { return __fadd_rn(acc[q].x, acc[q].y); };
        if (GEO) {
          const float tot = warp_totals<kGradStride>(s_red[wib], lane, value);
          // sums 16 to 19: eight lanes each, one 16-byte load per lane
          const float4 c = *reinterpret_cast<const float4*>(
              &s_red[wib][((lane >> 2) & 1) * red_upper(kGradStride) + (16 + (lane >> 3)) * kRedStride + 4 * (lane & 3)]);
          float rest = __fadd_rn(__fadd_rn(c.x, c.y), __fadd_rn(c.z, c.w));
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) rest = __fadd_rn(rest, __shfl_xor_sync(kFull, rest, o));
          if (lane < 16) sums[lane] = tot * red_sign;
          if ((lane & 7) == 0) sums[16 + (lane >> 3)] = rest;
        } else {
          const float tot = warp_totals<kRedSums>(s_red[wib], lane, [&](int q) { return value(red_target(q)); });
          if (lane < kRedSums) sums[red_dst] = tot * red_sign;
        }
        __syncwarp();  // the rows are read before the next entry writes them
      }
      // flush the batch: complete the centre gradient, then one vector atomic per
      // 4 slots and entry for the warp
      __syncwarp();
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int e = r * 32 + lane;
        if (e < cnt) {
          float* rs = &s_grad[wib][e * kGradStride];
          // dL/dc = -2 x the filter sums, minus the totals of dL/du, dL/dv and dL/dden times
          // the coefficients with which x - c enters u, v and den (g1.x, g1.z, g2.y for the
          // x offset; g1.y, g1.w, g2.z for y); the e0 slot holds the dL/dden total
          const float4 g1 = s_g1[wib][e], g2 = s_g2[wib][e];
          const float su = rs[kSumU], sv = rs[kSumV], se = rs[kGe0];
          rs[kGcx] = -2.f * rs[kGcx] - g2.y * se - g1.z * sv - g1.x * su;
          rs[kGcy] = -2.f * rs[kGcy] - g2.z * se - g1.w * sv - g1.y * su;
          rs[kSumU] = 0.f;
          rs[kSumV] = 0.f;
          float4* row = reinterpret_cast<float4*>(rs);
          float4* dst = reinterpret_cast<float4*>(a.grad_rec + (size_t)s_idx[wib][e] * kGradStride);
#pragma unroll
          for (int q = 0; q < kGradStride / 4; ++q) {
            const float4 g4 = row[q];
            if (g4.x != 0.f || g4.y != 0.f || g4.z != 0.f || g4.w != 0.f) {
              atomicAdd(dst + q, g4);
              row[q] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
        }
      }
    }
  }
}

template <int TW, int TH, int PPT, int BATCH>
cudaError_t bwd_dispatch(const RasterBwdArgs& a, cudaStream_t s) {
  const unsigned grid = warp_grid<TW, TH, PPT, kBW>(a.persistent_ctas, a.n_tiles);
  if (grid == 0) return cudaSuccess;
  if (a.d_out.depth || a.d_out.normal || a.d_out.depth2)
    raster_bwd_kernel<TW, TH, PPT, BATCH, true><<<grid, kBW * 32, 0, s>>>(a);
  else raster_bwd_kernel<TW, TH, PPT, BATCH, false><<<grid, kBW * 32, 0, s>>>(a);
  return launched();
}

}  // namespace

#ifdef OCGS_COUNT
extern "C" int ocgs_diag_read_bwd(unsigned long long* out, int reset) {
  cudaMemcpyFromSymbol(out, g_diag, sizeof(g_diag));
  if (reset) {
    unsigned long long z[2] = {0};
    cudaMemcpyToSymbol(g_diag, z, sizeof(z));
  }
  return 0;
}
#endif

cudaError_t launch_raster_backward(const RasterBwdArgs& a, int tile_w, int tile_h, int ppt, int batch,
                                   cudaStream_t s) {
#define OCGS_BWD(W, H, K, BT) \
  if (tile_w == W && tile_h == H && ppt == K && batch == BT) return bwd_dispatch<W, H, K, BT>(a, s);
  OCGS_RASTER_SHAPES(OCGS_BWD)
#undef OCGS_BWD
  return cudaErrorInvalidValue;
}

}  // namespace ocgs
