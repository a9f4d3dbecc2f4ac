// Map-accuracy metrics (Sec. IV measures a map by the PSNR and SSIM of its rendered views
// against the key-frames): per-image PSNR and SSIM of float images [B, C, H, W].
//
// PSNR = 10 log10(R^2 / MSE) over all C*H*W values of an image. SSIM (Wang et al. 2004) uses
// an 11 x 11 separable Gaussian window (sigma 1.5, taps normalised to sum 1) over zero-padded
// planes and C1 = (0.01 R)^2, C2 = (0.03 R)^2; an image's SSIM is the mean of its map.
//
// Both are deterministic: every block writes one partial sum to the caller's scratch, and one
// block per image adds its partials in a fixed order (in FP64). SSIM walks down a strip of columns,
// one column per thread: the five moments (x, y, x^2, y^2, xy) filtered along x are formed per row
// from a staged row group, and the last 11 rows of them, in registers, give the window sums.
#include <math.h>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kMetThreads = 256;
constexpr int kPsnrChunk = 8192;  // values per PSNR block
constexpr int kSsimTaps = 11;
constexpr int kSsimRad = kSsimTaps / 2;

struct Window {
  float w[kSsimTaps];
};

// sum over the block's 256 threads in a fixed order (shuffle tree, then the 8 warp sums in order)
__device__ __forceinline__ float block_sum(float v, float* s_warp) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.0f;
  if (threadIdx.x == 0)
    for (int w = 0; w < kMetThreads / 32; ++w) t += s_warp[w];
  return t;
}

__device__ __forceinline__ double block_sum_f64(double v, double* s_warp) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kMetThreads / 32; ++w) t += s_warp[w];
  return t;
}

__global__ void __launch_bounds__(kMetThreads) k_sqdiff(const float* __restrict__ x, const float* __restrict__ y,
                                                       int64_t per_image, int blocks_per_image,
                                                       float* __restrict__ partials) {
  pdl_begin();
  __shared__ float s_warp[kMetThreads / 32];
  const int64_t base = static_cast<int64_t>(blockIdx.y) * per_image;
  const int64_t lo = static_cast<int64_t>(blockIdx.x) * kPsnrChunk;
  const int64_t hi = lo + kPsnrChunk < per_image ? lo + kPsnrChunk : per_image;
  float acc = 0.0f;
  for (int64_t i = lo + threadIdx.x; i < hi; i += kMetThreads) {
    const float d = x[base + i] - y[base + i];
    acc = fmaf(d, d, acc);
  }
  const float t = block_sum(acc, s_warp);
  if (threadIdx.x == 0) partials[static_cast<int64_t>(blockIdx.y) * blocks_per_image + blockIdx.x] = t;
}

__global__ void __launch_bounds__(kMetThreads) k_psnr_final(const float* __restrict__ partials, int blocks_per_image,
                                                           int64_t per_image, float range, float* __restrict__ out) {
  pdl_begin();
  __shared__ double s_warp[kMetThreads / 32];
  double acc = 0.0;
  for (int j = threadIdx.x; j < blocks_per_image; j += kMetThreads)
    acc += partials[static_cast<int64_t>(blockIdx.x) * blocks_per_image + j];
  const double t = block_sum_f64(acc, s_warp);
  if (threadIdx.x == 0) {
    const double mse = t / static_cast<double>(per_image);
    const double r = range;
    out[blockIdx.x] = mse > 0.0 ? static_cast<float>(10.0 * log10(r * r / mse)) : INFINITY;
  }
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool in) {  // zero when !in
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(in ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One block per (strip of kSsimCols columns x kSsimRows rows, plane); plane = image * C + channel. Thread c
// owns output column c of the strip and keeps the five x-filtered moments of the last 11 input rows
// in registers; a group of 11 input rows is staged as (x, y) pairs at a time, so the loop over a group is
// unrolled and every register index is a constant. Bound by FP32 issue: 11 taps of 5 moments along x
// and along y per output, two moments per packed instruction. The 16 x 16 tile with shared x-filtered
// moments it replaces read 90 shared-memory words per output (27 here) and was bound by them: four
// 672x376 RGB images (both launches) 62 -> 33 us, eight 1280x720 ones 399 -> 167. 34 rows per strip
// (more blocks, more warm-up): 38 and 179; 128 columns: 38 and 160.
constexpr int kSsimCols = 64;
constexpr int kSsimRows = 45;  // output rows per strip: five groups of 11 input rows, less 10 of warm-up
constexpr int kSsimGroups = (kSsimRows + 2 * kSsimRad) / kSsimTaps;
static_assert(kSsimGroups * kSsimTaps == kSsimRows + 2 * kSsimRad, "whole groups of input rows");

__global__ void __launch_bounds__(kSsimCols) k_ssim(const float* __restrict__ x, const float* __restrict__ y, int H,
                                                    int W, int strips_x, int strips_per_plane, Window win, float c1,
                                                    float c2, float* __restrict__ map, float* __restrict__ partials) {
  pdl_begin();
  constexpr int kIn = kSsimCols + 2 * kSsimRad;
  __shared__ float2 s_in[2][kSsimTaps][kIn];
  __shared__ float s_warp[kSsimCols / 32];
  const int64_t plane = blockIdx.y;
  const int t = blockIdx.x, col = threadIdx.x;
  const int y0 = (t / strips_x) * kSsimRows, x0 = (t % strips_x) * kSsimCols;
  const int64_t HW = static_cast<int64_t>(H) * W;
  const float* xp = x + plane * HW;
  const float* yp = y + plane * HW;
  const int gx = x0 + col;
  // Group grp's rows go to buffer grp & 1 by asynchronous copies (zeros outside the image), which run
  // while the group before is filtered: a thread copies its own column, two threads per row the halo.
  const uint32_t smem0 = static_cast<uint32_t>(__cvta_generic_to_shared(&s_in[0][0][0]));
  auto copy = [&](int buf, int r, int c, int iy) {
    const int ix = x0 + c - kSsimRad;
    const bool in = iy >= 0 && iy < H && ix >= 0 && ix < W;
    const int64_t o = in ? static_cast<int64_t>(iy) * W + ix : 0;
    const uint32_t dst = smem0 + static_cast<uint32_t>(((buf * kSsimTaps + r) * kIn + c) * sizeof(float2));
    cp_async4(dst, xp + o, in);
    cp_async4(dst + 4, yp + o, in);
  };
  auto stage = [&](int grp) {
    const int iy0 = y0 + grp * kSsimTaps - kSsimRad;
#pragma unroll
    for (int r = 0; r < kSsimTaps; ++r) copy(grp & 1, r, col, iy0 + r);
    for (int i = col; i < 2 * kSsimRad * kSsimTaps; i += kSsimCols) {
      const int r = i / (2 * kSsimRad);
      copy(grp & 1, r, kSsimCols + i - r * 2 * kSsimRad, iy0 + r);
    }
  };
  float2 hm[kSsimTaps], hq[kSsimTaps];  // x-filtered (x, y) and (x^2, y^2) of input row r, at r % 11
  float hc[kSsimTaps];                  // and xy
  float tot = 0.0f;
  stage(0);
  for (int grp = 0; grp < kSsimGroups; ++grp) {
    cp_async_wait_all();
    __syncthreads();
    if (grp + 1 < kSsimGroups && y0 + (grp + 1) * kSsimTaps - kSsimRad < H + kSsimRad) stage(grp + 1);
#pragma unroll
    for (int r = 0; r < kSsimTaps; ++r) {
      float2 m = make_float2(0.0f, 0.0f), q = make_float2(0.0f, 0.0f);
      float c = 0.0f;
#pragma unroll
      for (int a = 0; a < kSsimTaps; ++a) {
        const float2 u = s_in[grp & 1][r][col + a];
        const float2 w = make_float2(win.w[a], win.w[a]);
        m = __ffma2_rn(w, u, m);
        q = __ffma2_rn(w, __fmul2_rn(u, u), q);
        c = fmaf(win.w[a], u.x * u.y, c);
      }
      hm[r] = m;
      hq[r] = q;
      hc[r] = c;
      // the window of output row gy ends at this input row; its first row is the oldest kept
      const int gy = y0 + grp * kSsimTaps + r - 2 * kSsimRad;
      if (grp * kSsimTaps + r < 2 * kSsimRad || gy >= H) continue;
      float2 mu = make_float2(0.0f, 0.0f), e2 = make_float2(0.0f, 0.0f);
      float exy = 0.0f;
#pragma unroll
      for (int a = 0; a < kSsimTaps; ++a) {
        const int s = (r + 1 + a) % kSsimTaps;
        const float2 w = make_float2(win.w[a], win.w[a]);
        mu = __ffma2_rn(w, hm[s], mu);
        e2 = __ffma2_rn(w, hq[s], e2);
        exy = fmaf(win.w[a], hc[s], exy);
      }
      const float mx = mu.x, my = mu.y;
      const float vx = e2.x - mx * mx, vy = e2.y - my * my, cxy = exy - mx * my;
      const float s = ((2.0f * mx * my + c1) * (2.0f * cxy + c2)) / ((mx * mx + my * my + c1) * (vx + vy + c2));
      if (gx < W) {
        if (map) map[plane * HW + static_cast<int64_t>(gy) * W + gx] = s;
        tot += s;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
  if ((col & 31) == 0) s_warp[col >> 5] = tot;
  __syncthreads();
  if (col == 0) {
    float sum = 0.0f;
#pragma unroll
    for (int w = 0; w < kSsimCols / 32; ++w) sum += s_warp[w];
    partials[plane * strips_per_plane + t] = sum;
  }
}

__global__ void __launch_bounds__(kMetThreads) k_mean_final(const float* __restrict__ partials, int64_t per_image,
                                                           double count, float* __restrict__ out) {
  pdl_begin();
  __shared__ double s_warp[kMetThreads / 32];
  double acc = 0.0;
  for (int64_t j = threadIdx.x; j < per_image; j += kMetThreads)
    acc += partials[static_cast<int64_t>(blockIdx.x) * per_image + j];
  const double t = block_sum_f64(acc, s_warp);
  if (threadIdx.x == 0) out[blockIdx.x] = static_cast<float>(t / count);
}

bool dims_ok(int32_t B, int32_t C, int32_t H, int32_t W) {
  return B >= 1 && C >= 1 && H >= 1 && W >= 1 && B <= 65535 && static_cast<int64_t>(B) * C <= 65535 && H <= 65536 &&
         W <= 65536;
}
int64_t psnr_blocks(int32_t C, int32_t H, int32_t W) {
  const int64_t n = static_cast<int64_t>(C) * H * W;
  return (n + kPsnrChunk - 1) / kPsnrChunk;
}
int64_t ssim_strips(int32_t H, int32_t W) {
  return static_cast<int64_t>((W + kSsimCols - 1) / kSsimCols) * ((H + kSsimRows - 1) / kSsimRows);
}
// Partial sums the scratch of gs_metrics_tmp_size holds per plane (one per 16 x 16 tile, of which a strip
// covers at least one).
int64_t ssim_scratch(int32_t H, int32_t W) {
  return static_cast<int64_t>((W + 15) / 16) * ((H + 15) / 16);
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" gs_status_t gs_metrics_tmp_size(int32_t images, int32_t channels, int32_t height, int32_t width,
                                           size_t* bytes) {
  if (!bytes || !dims_ok(images, channels, height, width)) return GS_ERR_INVALID_ARG;
  const int64_t a = images * psnr_blocks(channels, height, width);
  const int64_t b = static_cast<int64_t>(images) * channels * ssim_scratch(height, width);
  *bytes = static_cast<size_t>(a > b ? a : b) * sizeof(float);
  return GS_OK;
}

extern "C" gs_status_t gs_psnr(const float* x, const float* y, int32_t images, int32_t channels, int32_t height,
                               int32_t width, float data_range, float* psnr, void* tmp, size_t tmp_bytes,
                               void* stream) {
  size_t need = 0;
  if (!x || !y || !psnr || !tmp || !(data_range > 0.0f)) return GS_ERR_INVALID_ARG;
  if (gs_metrics_tmp_size(images, channels, height, width, &need) != GS_OK) return GS_ERR_INVALID_ARG;
  if (tmp_bytes < need) return GS_ERR_WORKSPACE_TOO_SMALL;
  const int64_t per_image = static_cast<int64_t>(channels) * height * width;
  const int nb = static_cast<int>(psnr_blocks(channels, height, width));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* part = static_cast<float*>(tmp);
  launch(k_sqdiff, dim3(nb, images), kMetThreads, 0, s, x, y, per_image, nb, part);
  launch(k_psnr_final, images, kMetThreads, 0, s, part, nb, per_image, data_range, psnr);
  return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}

extern "C" gs_status_t gs_ssim(const float* x, const float* y, int32_t images, int32_t channels, int32_t height,
                               int32_t width, float data_range, float* ssim, float* ssim_map, void* tmp,
                               size_t tmp_bytes, void* stream) {
  size_t need = 0;
  if (!x || !y || !ssim || !tmp || !(data_range > 0.0f)) return GS_ERR_INVALID_ARG;
  if (gs_metrics_tmp_size(images, channels, height, width, &need) != GS_OK) return GS_ERR_INVALID_ARG;
  if (tmp_bytes < need) return GS_ERR_WORKSPACE_TOO_SMALL;
  // normalised Gaussian taps, computed in FP64 and rounded once
  Window win;
  double w[kSsimTaps], sum = 0.0;
  for (int a = 0; a < kSsimTaps; ++a) {
    const double r = a - kSsimRad;
    w[a] = exp(-(r * r) / (2.0 * 1.5 * 1.5));
    sum += w[a];
  }
  for (int a = 0; a < kSsimTaps; ++a) win.w[a] = static_cast<float>(w[a] / sum);
  const float c1 = static_cast<float>((0.01 * data_range) * (0.01 * data_range));
  const float c2 = static_cast<float>((0.03 * data_range) * (0.03 * data_range));
  const int strips_x = (width + kSsimCols - 1) / kSsimCols;
  const int strips = static_cast<int>(ssim_strips(height, width));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* part = static_cast<float*>(tmp);
  launch(k_ssim, dim3(strips, images * channels), kSsimCols, 0, s, x, y, height, width, strips_x, strips, win, c1, c2,
         ssim_map, part);
  launch(k_mean_final, images, kMetThreads, 0, s, part, static_cast<int64_t>(channels) * strips,
         static_cast<double>(channels) * height * width, ssim);
  return cudaGetLastError() == cudaSuccess ? GS_OK : GS_ERR_CUDA;
}
