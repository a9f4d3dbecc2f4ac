// Forward compositing (gs_raster_fwd, gs_raster_fwd_stats, gs_raster_fwd_l1, and with the
// backward pass fused, gs_raster_fwd_l1_bwd); see raster_common.cuh for the staging and the
// opacity test both compositing kernels share.
#include <type_traits>

#include "raster_sweep.cuh"

namespace gs {
namespace {

// ============================================================================ forward
// A pixel that has stopped (or lies outside the image) moves to y = -inf: every later splat's exponent
// is then -inf (or not a number), so the pixel skips it without a separate flag. A kept splat that does not stop the pixel is blended
// through alpha, any other through 0, which leaves T and every accumulator bit for bit unchanged,
// so the blend needs no selects. STATS = true also counts the evaluations (list entries examined,
// including the one that stops a pixel) and the blended ones; the decisions and outputs are the same.
// L1 loss fused into the forward pass (LOSS = true): the targets, the gradient images it
// writes, per-tile partial sums and the block counter that elects the last block to finish,
// which sums the partials in tile order into *d_loss.
struct FusedLoss {
  const float* rgb_t;
  const float* depth_t;
  float* g_rgb;
  float* g_depth;
  float* partials;
  uint32_t* counter;
  float* d_loss;
};

__device__ __forceinline__ float sgn(float d) { return d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f); }

// Occlusion by an external surface (OCC = true): per pixel its depth and, optionally, colour
// ([K,H,W], [K,3,H,W]). The list is in depth order, so the first splat at or behind the surface
// ends the pixel (it is not composited); the surface then shows through the remaining
// transmittance: rgb += T ext_rgb, depth += T ext_depth.
struct Occlusion {
  const float* depth;
  const float* rgb;
};

// CHB > 0 (with LOSS only): the block continues into the backward pass of its tile (the sweep
// of gs_raster_bwd, staging CHB splats per chunk) as soon as its forward is done, from the loss
// gradient, colour, depth and last contributor of its pixels still in registers; the results
// equal gs_raster_fwd_l1 followed by gs_raster_bwd (dL_dT = NULL) with PX pixels per thread.
// The workspace is read-only to the forward; the variant with the fused backward also writes
// its gradient records, record bits and error word there, so it takes a mutable pointer.
template <int CHB>
using RasterWs = typename std::conditional<(CHB > 0), uint8_t*, const uint8_t*>::type;

// Shared memory of the forward: its staged chunk; with the fused backward, the backward sweep's
// shared memory in the same bytes (the forward's chunks are dead once every thread has passed
// the loss reduction's barriers, before the sweep starts).
template <int PX, int CH, int CHB, bool ROWS>
union FusedSmem {
  Stage<CH> S;
  BwdSmem<PX, CHB, ROWS> M;
};
template <int PX, int CH, int CHB, bool ROWS>
struct FwdSmemOf {
  using T = FusedSmem<PX, CH, CHB, ROWS>;
};
template <int PX, int CH, bool ROWS>
struct FwdSmemOf<PX, CH, 0, ROWS> {
  struct T {
    Stage<CH> S;
  };
};

// A thread's pixels against one splat. Minus the alpha with which each keeps it (0 where it doesn't) and
// whether it does; FULL evaluates the clamp and the power test too (see kChecked), OCC the occlusion.
template <int PX>
using Px = typename Vec<(PX >= 2 ? 2 : 1)>::T;
template <int PX, bool FULL, bool OCC>
__device__ __forceinline__ void pixel_alphas(const float4& A, const float4& B, Px<PX> npx,
                                             const Px<PX> (&npy)[PX >= 2 ? PX / 2 : 1], const float (&zmax)[PX],
                                             Px<PX> (&na)[PX >= 2 ? PX / 2 : 1], bool (&keep)[PX]) {
  constexpr int W = PX >= 2 ? 2 : 1, G = PX / W;
  const Column<W> col = splat_column<W>(A, B, npx);
  const Px<PX> Ay = bcast<W>(A.y);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const Px<PX> e = splat_exponent<W>(B, col, vadd(Ay, npy[g]));
#pragma unroll
    for (int i = 0; i < W; ++i) {
      const int q = g * W + i;
      const float raw = ex2_approx(comp(e, i));
      const float a = FULL ? fminf(raw, kAlphaMax) : raw;
      keep[q] = a >= kAlphaMin;
      if (FULL) keep[q] = keep[q] && comp(e, i) <= B.w;
      if (OCC) keep[q] = keep[q] && !(B.z >= zmax[q]);  // a splat at or behind the surface
      set_comp(na[g], i, keep[q] ? -a : 0.0f);
    }
  }
}
template <int PX>
__device__ __forceinline__ bool any_below(const Px<PX> (&t)[PX >= 2 ? PX / 2 : 1]) {
  constexpr int W = PX >= 2 ? 2 : 1;
  float low = comp(t[0], 0);
#pragma unroll
  for (int q = 1; q < PX; ++q) low = fminf(low, comp(t[q / W], q % W));
  return low < kTStop;
}
template <int PX>
__device__ __forceinline__ void blend(const float4& C, const Px<PX> (&na)[PX >= 2 ? PX / 2 : 1],
                                      const Px<PX> (&T)[PX >= 2 ? PX / 2 : 1], Px<PX> (&cr)[PX >= 2 ? PX / 2 : 1],
                                      Px<PX> (&cg)[PX >= 2 ? PX / 2 : 1], Px<PX> (&cb)[PX >= 2 ? PX / 2 : 1],
                                      Px<PX> (&cd)[PX >= 2 ? PX / 2 : 1]) {
  constexpr int W = PX >= 2 ? 2 : 1, G = PX / W;
  const Px<PX> nR = bcast<W>(C.x), nG = bcast<W>(C.y), nB = bcast<W>(C.z), nZ = bcast<W>(C.w);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const Px<PX> nw = vmul(na[g], T[g]);
    cr[g] = vfma(nR, nw, cr[g]);
    cg[g] = vfma(nG, nw, cg[g]);
    cb[g] = vfma(nB, nw, cb[g]);
    cd[g] = vfma(nZ, nw, cd[g]);
  }
}

// MANY = false (the fused variant only): compiled without the blocks-per-SM register budget, for
// grids that fit on the GPU in one wave anyway, where each block's own latency sets the time.
template <int PX, int CH, bool STATS, bool LOSS, bool OCC = false, int CHB = 0, bool MANY = true>
__global__ void __launch_bounds__(kTilePixels / PX,
                                  PX == 4 && MANY ? (CHB > 0 ? kMinBlocksFusedPx4 : kMinBlocksPx4)
                                                  : (PX == 2 && CHB > 0 ? kMinBlocksBwdPx2 : 1))
    k_raster_fwd(Layout L, RasterWs<CHB> __restrict__ ws, float* __restrict__ out_rgb, float* __restrict__ out_depth,
                 float* __restrict__ out_T, int32_t* __restrict__ out_last, uint64_t* __restrict__ evals_out,
                 uint64_t* __restrict__ blended_out, FusedLoss F, Occlusion O) {
  static_assert(CHB == 0 || (LOSS && !STATS && !OCC), "the fused backward follows the loss-fused forward");
  pdl_wait();
  constexpr int kThreads = kTilePixels / PX;
  constexpr int kWarps = kThreads / 32;
  // Two splats per turn (splat2): a warp waits less for its own chain of loads, exponentials and votes, and the
  // vote and the loop are paid once for two. Forward at 2 / 4 pixels, us: 300 tiles 28.6 -> 26.5 / 36.8 -> 30.7,
  // 3600 uneven 111 -> 107 / 126 -> 114, 9600 235 -> 225 / 201 -> 187, 57600 1547 -> 1475 / 1343 -> 1270; fused at 2
  // pixels 2 to 6%. Not in the fused kernel under the blocks-per-SM register budget (spills: 3.84 -> 3.88 ms).
  constexpr bool kPairs = !OCC && !STATS && PX >= 2 && !(CHB > 0 && PX == 4 && MANY);
  const float kInf = __int_as_float(0x7f800000);
  constexpr bool kRows = PX == 2 || (PX == 4 && !MANY);  // (see warp_reduce10_rows)
  __shared__ typename FwdSmemOf<PX, CH, CHB, kRows>::T sm;
  Stage<CH>& S = sm.S;
  __shared__ uint32_t s_red[2][kWarps];
  const TileCoord tc = tile_coord(L, blockIdx.x);
  const int lx = threadIdx.x & (kTile - 1), ly = (threadIdx.x / kTile) * PX;
  const int px = tc.tx * kTile + lx, py = tc.ty * kTile + ly;
  const uint64_t* keys = at<uint64_t>(ws, L.sorted ? L.keys[1] : L.keys[0]);
  const uint2 rg = at<uint2>(ws, L.ranges)[blockIdx.x];
  const float ox = static_cast<float>(tc.tx * kTile), oy = static_cast<float>(tc.ty * kTile);
  const float pxc = static_cast<float>(lx) + 0.5f, pyc = static_cast<float>(ly) + 0.5f;
  // this warp's pixel rows: (2 * warp) * PX .. (2 * warp + 2) * PX - 1
  const uint32_t wrows = ((1u << (2 * PX)) - 1u) << ((threadIdx.x >> 5) * 2 * PX);
  constexpr int W = PX >= 2 ? 2 : 1, G = PX / W;  // pixel q is component q % W of group q / W
  using V = typename Vec<W>::T;
  V T[G], cr[G], cg[G], cb[G], cd[G], npy[G];
  int32_t last[PX], stop_at[PX];
  float zmax[PX];
  uint32_t blended = 0;
  bool all_done = true;
  const V npx = bcast<W>(-pxc), one = bcast<W>(1.0f), zero = bcast<W>(0.0f);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    T[g] = one;
    cr[g] = cg[g] = cb[g] = cd[g] = zero;
#pragma unroll
    for (int i = 0; i < W; ++i) set_comp(npy[g], i, -(pyc + static_cast<float>(g * W + i)));
  }
#pragma unroll
  for (int q = 0; q < PX; ++q) {
    last[q] = 0;
    stop_at[q] = -1;
    const bool outside = !(px < L.W && py + q < L.H);
    if (outside) set_comp(npy[q / W], q % W, kInf);
    zmax[q] = kInf;
    if (OCC && !outside) zmax[q] = O.depth[tc.k * static_cast<int64_t>(L.H) * L.W + static_cast<int64_t>(py + q) * L.W + px];
    all_done = all_done && outside;
  }
  // the loss targets of the thread's pixels, loaded now so that the loads overlap the compositing
  float tgt[LOSS ? PX : 1][4];
  if (LOSS) {
    const int64_t HW = static_cast<int64_t>(L.H) * L.W;
#pragma unroll
    for (int q = 0; q < PX; ++q) {
      tgt[q][0] = tgt[q][1] = tgt[q][2] = tgt[q][3] = 0.0f;
      if (px < L.W && py + q < L.H) {
        const int64_t pix = static_cast<int64_t>(py + q) * L.W + px;
        const int64_t c0 = static_cast<int64_t>(tc.k) * 3 * HW + pix;
        tgt[q][0] = __ldg(F.rgb_t + c0);
        tgt[q][1] = __ldg(F.rgb_t + c0 + HW);
        tgt[q][2] = __ldg(F.rgb_t + c0 + 2 * HW);
        tgt[q][3] = __ldg(F.depth_t + tc.k * HW + pix);
      }
    }
  }
  // One splat of the staged chunk (list position pos): FULL evaluates the clamp and the power test
  // too (and the occlusion). The blend works on
  // -alpha (na) and the staged negated colours: T (1 - alpha) = fma(T, na, T) and c alpha T =
  // (-c)(na T) are the same roundings as with positive operands, without a negated copy of T.
  const int lane = threadIdx.x & 31;
  auto splat = [&](auto full, int j, int pos) {
    const float4 A = S.A[j], B = S.B[j], C = S.C[j];
    V na[G], Tn[G];
    bool keep[PX];
    pixel_alphas<PX, decltype(full)::value, OCC>(A, B, npx, npy, zmax, na, keep);
#pragma unroll
    for (int g = 0; g < G; ++g) Tn[g] = vfma(T[g], na[g], T[g]);
    // a pixel stops before the splat that would leave T < 1e-4 (once per pixel, so the changes are
    // made in a warp-uniform branch; a skipped splat leaves T, which is never below 1e-4)
    bool event = any_below<PX>(Tn);
    if (OCC) {
#pragma unroll
      for (int q = 0; q < PX; ++q) event = event || (B.z >= zmax[q] && comp(npy[q / W], q % W) != kInf);
    }
    if (__any_sync(0xffffffffu, event)) {
#pragma unroll
      for (int q = 0; q < PX; ++q) {
        const bool stop = comp(Tn[q / W], q % W) < kTStop;
        keep[q] = keep[q] && !stop;
        set_comp(na[q / W], q % W, stop ? 0.0f : comp(na[q / W], q % W));
        set_comp(npy[q / W], q % W, stop || (OCC && B.z >= zmax[q]) ? kInf : comp(npy[q / W], q % W));
        if (STATS) stop_at[q] = stop ? pos : stop_at[q];
      }
#pragma unroll
      for (int g = 0; g < G; ++g) Tn[g] = vfma(T[g], na[g], T[g]);
    }
    blend<PX>(C, na, T, cr, cg, cb, cd);
#pragma unroll
    for (int g = 0; g < G; ++g) T[g] = Tn[g];
#pragma unroll
    for (int q = 0; q < PX; ++q) {
      last[q] = keep[q] ? pos + 1 : last[q];
      if (STATS) blended += keep[q] ? 1u : 0u;
    }
  };
  auto all_stopped = [&]() -> bool {
    all_done = true;
#pragma unroll
    for (int q = 0; q < PX; ++q) all_done = all_done && comp(npy[q / W], q % W) == kInf;
    return __all_sync(0xffffffffu, all_done);
  };
  // Two successive splats of the warp's list (j0 before j1), bit for bit as one after the other: their
  // opacities don't depend on each other, so that the two chains of loads, exponentials and tests overlap, and
  // one vote serves both (T only falls, so a pixel that stops at either has the second T below 1e-4).
  auto splat2 = [&](auto full, int j0, int j1, int pos) {
    const float4 A0 = S.A[j0], B0 = S.B[j0], A1 = S.A[j1], B1 = S.B[j1];
    V n0[G], n1[G], T1[G], T2[G];
    bool keep0[PX], keep1[PX];
    pixel_alphas<PX, decltype(full)::value, OCC>(A0, B0, npx, npy, zmax, n0, keep0);
    pixel_alphas<PX, decltype(full)::value, OCC>(A1, B1, npx, npy, zmax, n1, keep1);
#pragma unroll
    for (int g = 0; g < G; ++g) {
      T1[g] = vfma(T[g], n0[g], T[g]);
      T2[g] = vfma(T1[g], n1[g], T1[g]);
    }
    if (__any_sync(0xffffffffu, any_below<PX>(T2))) {
#pragma unroll
      for (int q = 0; q < PX; ++q) {
        const bool stop = comp(T1[q / W], q % W) < kTStop;
        keep0[q] = keep0[q] && !stop;
        keep1[q] = keep1[q] && !stop;
        set_comp(n0[q / W], q % W, stop ? 0.0f : comp(n0[q / W], q % W));
        set_comp(n1[q / W], q % W, stop ? 0.0f : comp(n1[q / W], q % W));
        set_comp(npy[q / W], q % W, stop ? kInf : comp(npy[q / W], q % W));
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        T1[g] = vfma(T[g], n0[g], T[g]);
        T2[g] = vfma(T1[g], n1[g], T1[g]);
      }
#pragma unroll
      for (int q = 0; q < PX; ++q) {
        const bool stop = comp(T2[q / W], q % W) < kTStop;
        keep1[q] = keep1[q] && !stop;
        set_comp(n1[q / W], q % W, stop ? 0.0f : comp(n1[q / W], q % W));
        set_comp(npy[q / W], q % W, stop ? kInf : comp(npy[q / W], q % W));
      }
#pragma unroll
      for (int g = 0; g < G; ++g) T2[g] = vfma(T1[g], n1[g], T1[g]);
    }
    blend<PX>(S.C[j0], n0, T, cr, cg, cb, cd);
    blend<PX>(S.C[j1], n1, T1, cr, cg, cb, cd);
#pragma unroll
    for (int g = 0; g < G; ++g) T[g] = T2[g];
#pragma unroll
    for (int q = 0; q < PX; ++q) {
      last[q] = keep0[q] ? pos + j0 + 1 : last[q];
      last[q] = keep1[q] ? pos + j1 + 1 : last[q];
    }
  };
  for (uint32_t base = rg.x; base < rg.y; base += CH) {
    if (__syncthreads_count(!all_done) == 0) break;
    for (int jj = threadIdx.x; jj < CH; jj += kThreads) {
      const uint32_t i = base + jj;
      if (i < rg.y) stage_splat(S, jj, L, ws, keys, i, tc.k, ox, oy);
    }
    __syncthreads();
    const int n = min(CH, static_cast<int>(rg.y - base));
    const int pos0 = static_cast<int>(base - rg.x);
    // the splats that meet the warp's rows, 32 at a time (the loop runs over the set bits only; it
    // ends early when every pixel of the warp has stopped, looked at now and then)
    bool done = __all_sync(0xffffffffu, all_done);
#pragma unroll 1
    for (int w0 = 0; w0 < n && !done; w0 += 32) {
      const uint32_t r = w0 + lane < n ? S.rows[w0 + lane] : 0u;
      uint32_t visit = __ballot_sync(0xffffffffu, (r & wrows) != 0);
      const uint32_t checked = __ballot_sync(0xffffffffu, (r & kChecked) != 0);
      if constexpr (kPairs) {  // (a check every four turns, about every eight splats)
        int j = __ffs(visit) - 1;
#pragma unroll 1
        for (int turn = 1; j >= 0; ++turn) {
          visit &= visit - 1;
          int next = __ffs(visit) - 1;  // (found ahead of the splat's own chain)
          if (next >= 0) {
            visit &= visit - 1;
            const int after = __ffs(visit) - 1;
            if (((checked >> j) | (checked >> next)) & 1u) splat2(std::true_type{}, w0 + j, w0 + next, pos0);
            else splat2(std::false_type{}, w0 + j, w0 + next, pos0);
            next = after;
          } else if ((checked >> j) & 1u) {
            splat(std::true_type{}, w0 + j, pos0 + w0 + j);
          } else {
            splat(std::false_type{}, w0 + j, pos0 + w0 + j);
          }
          j = next;
          if ((turn & 3) == 0 && all_stopped()) break;
        }
        done = all_stopped();
      } else {  // (a check every eight list positions)
#pragma unroll 1
        for (int k = 0; visit && !done; k += 8) {
          uint32_t v = visit & (0xffu << k);
          visit &= ~(0xffu << k);
          int j = __ffs(v) - 1;
#pragma unroll 1
          while (j >= 0) {
            v &= v - 1;
            const int next = __ffs(v) - 1;
            if (OCC || ((checked >> j) & 1u)) splat(std::true_type{}, w0 + j, pos0 + w0 + j);
            else splat(std::false_type{}, w0 + j, pos0 + w0 + j);
            j = next;
          }
          done = all_stopped();
        }
      }
    }
  }
  if (CHB == 0) pdl_trigger();  // (the fused backward lets the next grid launch only at its end)
  const int64_t HW = static_cast<int64_t>(L.H) * L.W;
  const int len = static_cast<int>(rg.y - rg.x);
  float bg[CHB > 0 ? PX : 1][4];  // the loss gradient of each pixel (fused backward)
#pragma unroll
  for (int q = 0; q < (CHB > 0 ? PX : 1); ++q) bg[q][0] = bg[q][1] = bg[q][2] = bg[q][3] = 0.0f;
  uint32_t evals = 0;
  float loss = 0.0f;
  const float inv3 = 1.0f / (3.0f * static_cast<float>(HW));
  const float invd = L.lambda_depth / static_cast<float>(HW);
#pragma unroll
  for (int q = 0; q < PX; ++q) {
    const int y = py + q;
    float vr = comp(cr[q / W], q % W), vg = comp(cg[q / W], q % W), vb = comp(cb[q / W], q % W);
    float vd = comp(cd[q / W], q % W);
    const float vT = comp(T[q / W], q % W);
    if (px < L.W && y < L.H) {
      if (STATS) evals += static_cast<uint32_t>(stop_at[q] >= 0 ? stop_at[q] + 1 : len);
      const int64_t pix = static_cast<int64_t>(y) * L.W + px;
      const int64_t c0 = static_cast<int64_t>(tc.k) * 3 * HW + pix;
      if (OCC) {  // the external surface through the remaining transmittance
        if (O.rgb) {
          vr = __fmaf_rn(vT, O.rgb[c0], vr);
          vg = __fmaf_rn(vT, O.rgb[c0 + HW], vg);
          vb = __fmaf_rn(vT, O.rgb[c0 + 2 * HW], vb);
        }
        vd = __fmaf_rn(vT, zmax[q], vd);
      }
      if (out_rgb) {
        out_rgb[c0] = vr;
        out_rgb[c0 + HW] = vg;
        out_rgb[c0 + 2 * HW] = vb;
      }
      if (out_depth) out_depth[tc.k * HW + pix] = vd;
      if (out_T) out_T[tc.k * HW + pix] = vT;
      if (out_last) out_last[tc.k * HW + pix] = last[q];
      if (LOSS) {
        // L = sum_k [ mean_{3HW} |R - R*| + lambda mean_{HW} |D - D*| ], sign(0) = 0
        const float c[3] = {vr, vg, vb};
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) {
          const float d = c[ch] - tgt[LOSS ? q : 0][ch];
          loss += fabsf(d) * inv3;
          const float gv = sgn(d) * inv3;
          F.g_rgb[c0 + ch * HW] = gv;
          if (CHB > 0) bg[CHB > 0 ? q : 0][ch] = gv;
        }
        const float d = vd - tgt[LOSS ? q : 0][3];
        loss += fabsf(d) * invd;
        const float gv = sgn(d) * invd;
        F.g_depth[tc.k * HW + pix] = gv;
        if (CHB > 0) bg[CHB > 0 ? q : 0][3] = gv;
      }
    }
  }
  if (LOSS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    __shared__ float s_loss[kWarps];
    __shared__ bool s_last;
    if ((threadIdx.x & 31) == 0) s_loss[threadIdx.x >> 5] = loss;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.0f;
      for (int w = 0; w < kWarps; ++w) t += s_loss[w];
      F.partials[blockIdx.x] = t;
      __threadfence();
      s_last = atomicAdd(F.counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (s_last) {
      // the last block sums every tile's partial in a fixed order
      __threadfence();
      float v = 0.0f;
      for (uint32_t i = threadIdx.x; i < gridDim.x; i += kThreads) v += __ldcg(&F.partials[i]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      __syncthreads();
      if ((threadIdx.x & 31) == 0) s_loss[threadIdx.x >> 5] = v;
      __syncthreads();
      if (threadIdx.x == 0) {
        float t = 0.0f;
        for (int w = 0; w < kWarps; ++w) t += s_loss[w];
        F.d_loss[0] = t;
        *F.counter = 0;
      }
    }
  }
  if constexpr (CHB > 0) {
    // the backward pass of this tile, from registers: the weighted colour behind the first
    // splat is the loss gradient applied to the pixel's output (no dL/dT_final term)
    BwdSmem<PX, CHB, kRows>& M = sm.M;
    float Sg[PX], hT[PX], gr[PX], gg[PX], gb[PX], gd[PX];
    int lst[PX];
#pragma unroll
    for (int q = 0; q < PX; ++q) {
      gr[q] = bg[q][0];
      gg[q] = bg[q][1];
      gb[q] = bg[q][2];
      gd[q] = bg[q][3];
      const bool in = px < L.W && py + q < L.H;
      Sg[q] = in ? weighted_colour(gr[q], gg[q], gb[q], gd[q], comp(cr[q / W], q % W), comp(cg[q / W], q % W),
                                   comp(cb[q / W], q % W), comp(cd[q / W], q % W))
                 : 0.0f;
      hT[q] = 0.0f;
      lst[q] = in ? last[q] : 0;
    }
    bwd_sweep<PX, CHB, false, kRows>(M, L, ws, tc, rg, Sg, hT, gr, gg, gb, gd, lst);
    pdl_trigger();
  }
  if (STATS) {
    uint32_t e = evals, c = blended;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) {
      s_red[0][threadIdx.x >> 5] = e;
      s_red[1][threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint64_t te = 0, tcn = 0;
      for (int w = 0; w < kWarps; ++w) {
        te += s_red[0][w];
        tcn += s_red[1][w];
      }
      if (te) atomicAdd(reinterpret_cast<unsigned long long*>(evals_out), static_cast<unsigned long long>(te));
      if (tcn) atomicAdd(reinterpret_cast<unsigned long long*>(blended_out), static_cast<unsigned long long>(tcn));
    }
  }
}

}  // namespace

cudaError_t launch_raster_fwd_l1_bwd(const Layout& L, void* ws, float* rgb, float* depth, float* T_final, int32_t* last,
                                     const FusedLossArgs& loss, cudaStream_t s) {
  Status* st = at<Status>(ws, L.status);
  if (L.n_tiles == 0) {
    cudaMemsetAsync(loss.d_loss, 0, sizeof(float), s);
    return cudaGetLastError();
  }
  const unsigned grid = static_cast<unsigned>(L.n_tiles);
  uint8_t* w = static_cast<uint8_t*>(ws);
  uint64_t *ev = &st->evals, *cp = &st->composited;
  const FusedLoss F{loss.rgb_t, loss.depth_t, loss.g_rgb, loss.g_depth, at<float>(ws, L.tile_loss), &st->loss_ctr,
                    loss.d_loss};
  const int px = pick_px(L.fwd_px, default_px(L));
  const int ch = pick_chunk(L.fwd_chunk, 64, 256, kFwdChunk);
  // the backward phase stages kBwdChunk splats per chunk (the chunk depth changes no result); at 4
  // pixels per thread, a grid that the variant without the blocks-per-SM register budget runs in
  // one wave (its resident blocks per SM, from the occupancy calculator, times the SMs) takes it
  static int uncapped_blocks[64] = {};  // per device: resident blocks per SM of the uncapped variant
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!uncapped_blocks[dev]) {
    int b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_raster_fwd<4, 128, false, true, false, kBwdChunk, false>,
                                                  kTilePixels / 4, 0);
    uncapped_blocks[dev] = b > 0 ? b : 1;
  }
  const bool one_wave = L.n_tiles <= static_cast<int64_t>(device_sms()) * uncapped_blocks[dev];
#define GS_FB_M(P, C, M)                                                                                             \
  launch(k_raster_fwd<P, C, false, true, false, kBwdChunk, M>, grid, kTilePixels / P,                                 \
         cap_smem(k_raster_fwd<P, C, false, true, false, kBwdChunk, M>, L.raster_bps), s, L, w, rgb, depth, T_final, \
         last, ev, cp, F, Occlusion{})
#define GS_FB(P, C)                       \
  if (one_wave) {                         \
    GS_FB_M(P, C, (P != 4));              \
  } else {                                \
    GS_FB_M(P, C, true);                  \
  }
#define GS_FB_CH(P)                  \
  switch (ch) {                      \
    case 64: GS_FB(P, 64); break;    \
    case 256: GS_FB(P, 256); break;  \
    default: GS_FB(P, 128); break;   \
  }
  switch (px) {
    case 1: GS_FB_CH(1); break;
    case 2: GS_FB_CH(2); break;
    default: GS_FB_CH(4); break;
  }
#undef GS_FB_CH
#undef GS_FB
#undef GS_FB_M
  return cudaGetLastError();
}

cudaError_t launch_raster_fwd(const Layout& L, void* ws, float* rgb, float* depth, float* T_final, int32_t* last,
                              bool stats, const FusedLossArgs* loss, cudaStream_t s, const float* ext_depth,
                              const float* ext_rgb) {
  Status* st = at<Status>(ws, L.status);
  if (stats) {
    cudaMemsetAsync(&st->evals, 0, sizeof(uint64_t), s);
    cudaMemsetAsync(&st->composited, 0, sizeof(uint64_t), s);
  }
  if (L.n_tiles == 0) {
    if (loss) cudaMemsetAsync(loss->d_loss, 0, sizeof(float), s);
    return cudaGetLastError();
  }
  const unsigned grid = static_cast<unsigned>(L.n_tiles);
  const uint8_t* w = static_cast<const uint8_t*>(ws);
  uint64_t *ev = &st->evals, *cp = &st->composited;
  FusedLoss F{};
  if (loss)
    F = FusedLoss{loss->rgb_t, loss->depth_t, loss->g_rgb, loss->g_depth, at<float>(ws, L.tile_loss), &st->loss_ctr,
                  loss->d_loss};
  const int px = pick_px(L.fwd_px, default_px(L));
  const int ch = pick_chunk(L.fwd_chunk, 64, 256, kFwdChunk);
#define GS_FWD(P, C, ST, LO)                                                                                  \
  launch(k_raster_fwd<P, C, ST, LO>, grid, kTilePixels / P, cap_smem(k_raster_fwd<P, C, ST, LO>, L.raster_bps), s, \
         L, w, rgb, depth, T_final, last, ev, cp, F, Occlusion{})
#define GS_FWD_CH(P, ST, LO)              \
  switch (ch) {                           \
    case 64: GS_FWD(P, 64, ST, LO); break;   \
    case 256: GS_FWD(P, 256, ST, LO); break; \
    default: GS_FWD(P, 128, ST, LO); break;  \
  }
  if (ext_depth) {  // occlusion by an external surface: one chunk depth
    const Occlusion O{ext_depth, ext_rgb};
    switch (px) {
      case 1: launch(k_raster_fwd<1, kFwdChunk, false, false, true>, grid, kTilePixels, 0, s, L, w, rgb, depth, T_final,
                     last, ev, cp, F, O); break;
      case 2: launch(k_raster_fwd<2, kFwdChunk, false, false, true>, grid, kTilePixels / 2, 0, s, L, w, rgb, depth,
                     T_final, last, ev, cp, F, O); break;
      default: launch(k_raster_fwd<4, kFwdChunk, false, false, true>, grid, kTilePixels / 4, 0, s, L, w, rgb, depth,
                      T_final, last, ev, cp, F, O); break;
    }
  } else if (stats) {  // the counting variant: one chunk depth (the chunking changes no decision)
    switch (px) {
      case 1: GS_FWD(1, kFwdChunk, true, false); break;
      case 2: GS_FWD(2, kFwdChunk, true, false); break;
      default: GS_FWD(4, kFwdChunk, true, false); break;
    }
  } else if (loss) {
    switch (px) {
      case 1: GS_FWD_CH(1, false, true); break;
      case 2: GS_FWD_CH(2, false, true); break;
      default: GS_FWD_CH(4, false, true); break;
    }
  } else {
    switch (px) {
      case 1: GS_FWD_CH(1, false, false); break;
      case 2: GS_FWD_CH(2, false, false); break;
      default: GS_FWD_CH(4, false, false); break;
    }
  }
#undef GS_FWD_CH
#undef GS_FWD
  return cudaGetLastError();
}

}  // namespace gs
