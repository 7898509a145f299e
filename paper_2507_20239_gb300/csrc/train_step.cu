// The rest of a training step around the rasterizer: the photometric loss of
// Eq. 3 with its gradient, (1 - lambda) L1 + lambda D-SSIM, and the optimiser
// update (Adam; sparse Adam skips Gaussians no view of the step saw), with the
// opacity reset of the densification schedule.
//
// SSIM: per channel, an 11 x 11 Gaussian window (sigma 1.5, normalised) applied
// separably with zero padding; mu_x, mu_y and the windowed second moments Sxx, Syy,
// Sxy give map = (2 mu_x mu_y + C1)(2 (Sxy - mu_x mu_y) + C2) /
// ((mu_x^2 + mu_y^2 + C1)(Sxx - mu_x^2 + Syy - mu_y^2 + C2)). Its gradient w.r.t. the
// rendered image x is the window's adjoint (the same symmetric window, zero
// padded) applied to d map / d mu_x, d map / d Sxx and d map / d Sxy, combined as
// W*(d/dmu) + 2 x W*(d/dSxx) + y W*(d/dSxy). Two kernels, every view of the frame in
// one launch each: the window sums and the map's derivatives, then their adjoint and the
// gradient; the sums for the loss are carried in FP32 pairs per thread and FP64 across.
#include <algorithm>
#include <cmath>

#include "gs_common.cuh"

namespace gs {

constexpr int kWin = 11, kHalf = 5;
constexpr float kSsimC1 = 0.01f * 0.01f, kSsimC2 = 0.03f * 0.03f;
constexpr int kPlanes = 3;   // scratch planes per pixel value: the map's derivatives

struct float5_t {
  float v[5];
};

// Both kernels take tiles of 64 x 22 output values. The inputs with their halo of 5 go to
// shared memory once; a thread then forms four adjacent horizontal window sums (14
// values read for 44 taps) into shared memory, and up to six vertical ones of a column
// (16 values for 66 taps) from there. Bound by FP32 issue: about 170 instructions a value
// in the first kernel, 100 in the second, pairs of moments packed (f32x2: the same
// operations and roundings at half the issue slots). One thread per value with every tap
// read from global memory, in four passes over eight planes, was bound by those
// loads: 3 x 826 x 1246 84 + 46 + 44 + 40 us and a finishing launch -> 37 + 27 us, the
// same bits. Walking down a strip with the last 11 rows' sums in registers came to 44 + 31
// us (128 registers: too few warps to cover the loads).
// 22 rows: 32 rows with the halo x 16 groups of four = two rounds of 256 threads.
constexpr int kTx = 64, kTy = 22, kSsimThreads = 256;
constexpr int kTileRows = kTy + 2 * kHalf, kTileCols = kTx + 2 * kHalf + 2;   // whole 16-byte pairs
constexpr int kColRows = (kTy + kSsimThreads / kTx - 1) / (kSsimThreads / kTx);   // output rows per thread
static_assert((kTileRows * kTx / 4) % kSsimThreads == 0, "whole rounds of horizontal tasks");

// Interleaved pairs are read and written four at a time, 32 bytes apart from thread to
// thread; swapping neighbouring 16-byte chunks in every other run of eight keeps those
// accesses off each other's banks. pair_at: the slot of column c of a row.
__device__ __forceinline__ int chunk_at(int chunk) { return chunk ^ ((chunk >> 3) & 1); }
__device__ __forceinline__ int pair_at(int c) { return chunk_at(c >> 1) * 2 + (c & 1); }

struct SsimTile {
  float2 in2[kTileRows][kTileCols + 4];   // two input planes, interleaved (rows of whole 16-chunk swaps)
  float2 h1[kTileRows][kTx];              // horizontal sums
  float2 h2[kTileRows][kTx];
  float h3[kTileRows][kTx];
};
struct GradTile {
  float2 in2[kTileRows][kTileCols + 4];
  float in1[kTileRows][kTileCols];    // the third plane
  float2 h1[kTileRows][kTx];
  float h3[kTileRows][kTx];
};
static_assert(kTileCols % 4 == 0, "16-byte aligned rows");

// The window's weights exp(-d^2 / (2 1.5^2)), d = -5 .. 5, for the block (a barrier follows).
__device__ __forceinline__ void put_window(float *w) {
  if (threadIdx.x < kWin) {
    const float d = (float)((int)threadIdx.x - kHalf);
    w[threadIdx.x] = expf(-d * d / (2.f * 1.5f * 1.5f));
  }
}
// The first six as pairs (the window is symmetric), and the inverse of the sum of all.
__device__ __forceinline__ float get_window(const float *w, float2 wr[kHalf + 1]) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kWin; ++k) s += w[k];
#pragma unroll
  for (int k = 0; k <= kHalf; ++k) wr[k] = f2(w[k]);
  return 1.f / s;
}

struct Tile {
  int W, H, x0, y0;   // the view's size, the tile's first column and row
  int64_t base;       // offset of this (view, channel) plane in the planar batch layout
  bool on;
};

__device__ __forceinline__ Tile tile_of(const gs_camera_t *cams) {
  Tile p;
  const int v = blockIdx.z / 3, c = blockIdx.z - 3 * v;
  const gs_camera_t &cam = cams[v];
  p.W = cam.width;
  p.H = cam.height;
  p.base = 3 * cam.pixel_offset + (int64_t)c * p.W * p.H;
  p.x0 = blockIdx.x * kTx;
  p.y0 = blockIdx.y * kTy;
  p.on = p.x0 < p.W && p.y0 < p.H;
  return p;
}

// The tile's inputs and their halo, zero outside the view: planes a and b interleaved and,
// with C, plane c.
template <bool C, typename T>
__device__ __forceinline__ void load_tile(const Tile &p, T &s, const float *__restrict__ a, const float *__restrict__ b,
                                          const float *__restrict__ c, float *s_c) {
  // a warp takes every eighth row, its lanes the columns lane, lane + 32, lane + 64
  constexpr int kWarps = kSsimThreads / 32, kCols = (kTileCols + 31) / 32;
  const int lane = threadIdx.x & 31;
  const int x = p.x0 - kHalf + lane;
#pragma unroll
  for (int r = threadIdx.x >> 5; r < kTileRows; r += kWarps) {
    const int y = p.y0 - kHalf + r;
    const bool row = (unsigned)y < (unsigned)p.H;
    const int64_t o = p.base + (int64_t)y * p.W + x;
#pragma unroll
    for (int q = 0; q < kCols; ++q) {
      const int col = lane + 32 * q;
      if (col >= kTileCols) break;
      float2 v = make_float2(0.f, 0.f);
      float u = 0.f;
      if (row && (unsigned)(x + 32 * q) < (unsigned)p.W) {
        v = make_float2(a[o + 32 * q], b[o + 32 * q]);
        if (C) u = c[o + 32 * q];
      }
      s.in2[r][pair_at(col)] = v;
      if (C) s_c[r * kTileCols + col] = u;
    }
  }
}

// The 14 interleaved values from column 4 g of row r.
__device__ __forceinline__ void read14(const float2 *row, int g, float2 v[14]) {
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const float4 f = *reinterpret_cast<const float4 *>(row + chunk_at(2 * g + q) * 2);
    v[2 * q] = make_float2(f.x, f.y);
    v[2 * q + 1] = make_float2(f.z, f.w);
  }
}

__device__ __forceinline__ void write4(float2 *row, int g, const float2 v[4]) {
  *reinterpret_cast<float4 *>(row + chunk_at(2 * g) * 2) = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
  *reinterpret_cast<float4 *>(row + chunk_at(2 * g + 1) * 2) = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
}

// Window sums of x, y, x^2, y^2, x y -> SSIM map (summed per view) and its partial
// derivatives w.r.t. mu_x, Sxx, Sxy (planes 0..2); L1 sum.
__global__ void __launch_bounds__(kSsimThreads, 3) ssim_map_kernel(
    const gs_camera_t *__restrict__ cams, const float *__restrict__ img, const float *__restrict__ tgt,
    float *__restrict__ ws, int64_t stride, double *l1, double *ssim_sum) {
  extern __shared__ float4 s_raw[];
  SsimTile &s = *reinterpret_cast<SsimTile *>(s_raw);
  __shared__ float w[kWin];
  __shared__ float4 s_red[kSsimThreads / 32];
  const Tile p = tile_of(cams);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float ad = 0.f, ad_c = 0.f, ms = 0.f, ms_c = 0.f;
  if (p.on) {
    put_window(w);
    load_tile<false>(p, s, img, tgt, nullptr, nullptr);
    __syncthreads();
    float2 wr[kHalf + 1];
    const float n = get_window(w, wr);
    for (int t = threadIdx.x; t < kTileRows * kTx / 4; t += kSsimThreads) {
      const int r = t / (kTx / 4), g = t - r * (kTx / 4);
      float2 v[14];
      read14(s.in2[r], g, v);
      float2 a1[4], a2[4];
      float a3[4];
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        a1[o] = a2[o] = f2(0.f);
        a3[o] = 0.f;
      }
#pragma unroll
      for (int c = 0; c < 14; ++c) {   // taps in ascending column order
        const float2 vv = f2_mul(v[c], v[c]);
        const float xy = __fmul_rn(v[c].x, v[c].y);
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int k = c - o;
          if (k < 0 || k >= kWin) continue;
          const float2 wk = wr[k <= kHalf ? k : kWin - 1 - k];
          a1[o] = f2_fma(wk, v[c], a1[o]);
          a2[o] = f2_fma(wk, vv, a2[o]);
          a3[o] = fmaf(wk.x, xy, a3[o]);
        }
      }
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        a1[o] = f2_mul(a1[o], f2(n));
        a2[o] = f2_mul(a2[o], f2(n));
        a3[o] *= n;
      }
      write4(s.h1[r], g, a1);
      write4(s.h2[r], g, a2);
      *reinterpret_cast<float4 *>(&s.h3[r][4 * g]) = make_float4(a3[0], a3[1], a3[2], a3[3]);
    }
    __syncthreads();
    const int c = threadIdx.x % kTx, r0 = (threadIdx.x / kTx) * kColRows;
    const int rows = min(kColRows, min(kTy, p.H - p.y0) - r0);
    if (p.x0 + c < p.W && rows > 0) {
      float2 b1[kColRows], b2[kColRows];
      float b3[kColRows];
#pragma unroll
      for (int o = 0; o < kColRows; ++o) {
        b1[o] = b2[o] = f2(0.f);
        b3[o] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < kColRows + 2 * kHalf; ++i) {   // taps in ascending row order
        if (r0 + i >= kTileRows) break;                  // past the tile: rows not kept
        const float2 h1 = s.h1[r0 + i][pair_at(c)], h2 = s.h2[r0 + i][pair_at(c)];
        const float h3 = s.h3[r0 + i][c];
#pragma unroll
        for (int o = 0; o < kColRows; ++o) {
          const int k = i - o;
          if (k < 0 || k >= kWin) continue;
          const float2 wk = wr[k <= kHalf ? k : kWin - 1 - k];
          b1[o] = f2_fma(wk, h1, b1[o]);
          b2[o] = f2_fma(wk, h2, b2[o]);
          b3[o] = fmaf(wk.x, h3, b3[o]);
        }
      }
#pragma unroll
      for (int o = 0; o < kColRows; ++o) {
        if (o >= rows) break;
        const float mx = b1[o].x * n, my = b1[o].y * n, sxx = b2[o].x * n, syy = b2[o].y * n, sxy = b3[o] * n;
        const float A1 = 2.f * mx * my + kSsimC1, A2 = 2.f * (sxy - mx * my) + kSsimC2;
        const float B1 = mx * mx + my * my + kSsimC1, B2 = (sxx - mx * mx) + (syy - my * my) + kSsimC2;
        const float inv = 1.f / (B1 * B2);
        const float mapv = A1 * A2 * inv;
        const int64_t i = p.base + (int64_t)(p.y0 + r0 + o) * p.W + p.x0 + c;
        ws[i] = (2.f * my * (A2 - A1)) * inv - mapv * (2.f * mx * (B2 - B1)) * inv;   // d map / d mu_x
        ws[stride + i] = -mapv / B2;                                                  // d map / d Sxx
        ws[2 * stride + i] = 2.f * A1 * inv;                                          // d map / d Sxy
        pair_add(ms, ms_c, mapv);
        const float2 v = s.in2[r0 + o + kHalf][pair_at(c + kHalf)];
        pair_add(ad, ad_c, fabsf(v.x - v.y));
      }
    }
  }
  warp_pair_sum(ad, ad_c);
  warp_pair_sum(ms, ms_c);
  if (lane == 0) s_red[warp] = make_float4(ad, ad_c, ms, ms_c);
  __syncthreads();
  if (warp == 0) {
    const float4 q = s_red[lane % (kSsimThreads / 32)];
    ad = q.x; ad_c = q.y; ms = q.z; ms_c = q.w;
    warp_pair_sum(ad, ad_c, kSsimThreads / 64);
    warp_pair_sum(ms, ms_c, kSsimThreads / 64);
  }
  if (threadIdx.x == 0) {
    const double da = (double)ad + (double)ad_c, dm = (double)ms + (double)ms_c;
    atomicAdd(l1 + blockIdx.z / 3, da);
    atomicAdd(ssim_sum + blockIdx.z / 3, dm);
  }
}

// Adjoint window sums of the derivative planes -> d loss / d image; the views' losses from
// the sums.
__global__ void __launch_bounds__(kSsimThreads, 3) ssim_grad_kernel(const gs_camera_t *__restrict__ cams,
                                                                    const float *__restrict__ img,
                                                                    const float *__restrict__ tgt,
                                                                    const float *__restrict__ ws, int64_t stride,
                                                                    float lambda, const double *__restrict__ l1,
                                                                    const double *__restrict__ ssim_sum,
                                                                    float *__restrict__ loss,
                                                                    float *__restrict__ d_image) {
  extern __shared__ float4 s_raw[];
  GradTile &s = *reinterpret_cast<GradTile *>(s_raw);
  __shared__ float w[kWin];
  const Tile p = tile_of(cams);
  if (!p.on) return;
  if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z % 3 == 0 && threadIdx.x == 0) {
    const int v = blockIdx.z / 3;
    const double cnt = 3.0 * p.W * (double)p.H;
    loss[v] = (float)((1.0 - lambda) * l1[v] / cnt + lambda * (1.0 - ssim_sum[v] / cnt));
  }
  put_window(w);
  load_tile<true>(p, s, ws, ws + stride, ws + 2 * stride, &s.in1[0][0]);
  __syncthreads();
  float2 wr[kHalf + 1];
  const float n = get_window(w, wr);
  for (int t = threadIdx.x; t < kTileRows * kTx / 4; t += kSsimThreads) {
    const int r = t / (kTx / 4), g = t - r * (kTx / 4);
    float2 v[14];
    read14(s.in2[r], g, v);
    float u[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 f = *reinterpret_cast<const float4 *>(&s.in1[r][4 * (g + q)]);
      u[4 * q] = f.x; u[4 * q + 1] = f.y; u[4 * q + 2] = f.z; u[4 * q + 3] = f.w;
    }
    float2 a1[4];
    float a3[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      a1[o] = f2(0.f);
      a3[o] = 0.f;
    }
#pragma unroll
    for (int c = 0; c < 14; ++c)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int k = c - o;
        if (k < 0 || k >= kWin) continue;
        const float2 wk = wr[k <= kHalf ? k : kWin - 1 - k];
        a1[o] = f2_fma(wk, v[c], a1[o]);
        a3[o] = fmaf(wk.x, u[c], a3[o]);
      }
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      a1[o] = f2_mul(a1[o], f2(n));
      a3[o] *= n;
    }
    write4(s.h1[r], g, a1);
    *reinterpret_cast<float4 *>(&s.h3[r][4 * g]) = make_float4(a3[0], a3[1], a3[2], a3[3]);
  }
  __syncthreads();
  const int c = threadIdx.x % kTx, r0 = (threadIdx.x / kTx) * kColRows;
  const int rows = min(kColRows, min(kTy, p.H - p.y0) - r0);
  if (p.x0 + c >= p.W || rows <= 0) return;
  const int64_t i0 = p.base + (int64_t)(p.y0 + r0) * p.W + p.x0 + c;
  float xs[kColRows], ys[kColRows];
#pragma unroll
  for (int o = 0; o < kColRows; ++o)
    if (o < rows) {
      xs[o] = img[i0 + (int64_t)o * p.W];
      ys[o] = tgt[i0 + (int64_t)o * p.W];
    }
  float2 b1[kColRows];
  float b3[kColRows];
#pragma unroll
  for (int o = 0; o < kColRows; ++o) {
    b1[o] = f2(0.f);
    b3[o] = 0.f;
  }
#pragma unroll
  for (int i = 0; i < kColRows + 2 * kHalf; ++i) {
    if (r0 + i >= kTileRows) break;
    const float2 h1 = s.h1[r0 + i][pair_at(c)];
    const float h3 = s.h3[r0 + i][c];
#pragma unroll
    for (int o = 0; o < kColRows; ++o) {
      const int k = i - o;
      if (k < 0 || k >= kWin) continue;
      const float2 wk = wr[k <= kHalf ? k : kWin - 1 - k];
      b1[o] = f2_fma(wk, h1, b1[o]);
      b3[o] = fmaf(wk.x, h3, b3[o]);
    }
  }
  const float inv_n = 1.f / (3.f * (float)p.W * (float)p.H);
#pragma unroll
  for (int o = 0; o < kColRows; ++o) {
    if (o >= rows) break;
    const float xi = xs[o], yi = ys[o], d = xi - yi;
    const float g_ssim = (b1[o].x * n + 2.f * xi * (b1[o].y * n) + yi * (b3[o] * n)) * inv_n;
    const float g_l1 = d > 0.f ? inv_n : (d < 0.f ? -inv_n : 0.f);
    d_image[i0 + (int64_t)o * p.W] = (1.f - lambda) * g_l1 - lambda * g_ssim;
  }
}

// ------------------------------------------------------------------ optimiser
// One parameter group's update, by the whole grid.
__device__ __forceinline__ void adam_group(int grp, const gs_params_out_t &P, const gs_param_grads_t &G,
                                           const gs_adam_state_t &S, int64_t n, int32_t sh_width, float ss, float beta1,
                                           float beta2, float eps, float sqrt_bc2, const int32_t *__restrict__ radius,
                                           int32_t n_views) {
  float *p;
  const float *g;
  int width;
  switch (grp) {
    case 0: p = P.means; g = G.d_means; width = 3; break;
    case 1: p = P.log_scales; g = G.d_log_scales; width = 3; break;
    case 2: p = P.quats; g = G.d_quats; width = 4; break;
    case 3: p = P.opacity_logits; g = G.d_opacity_logits; width = 1; break;
    default: p = P.sh; g = G.d_sh; width = sh_width; break;
  }
  float *m = S.m[grp], *v = S.v[grp];
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto visible = [&](int64_t row) {
    bool seen = false;
    for (int k = 0; k < n_views; ++k) seen |= radius[(int64_t)k * n + row] > 0;
    return seen;
  };
  auto update = [&](float &pi, float &mi, float &vi, float gi) {
    mi = beta1 * mi + (1.f - beta1) * gi;
    vi = beta2 * vi + (1.f - beta2) * gi * gi;
    pi -= ss * mi / (sqrtf(vi) / sqrt_bc2 + eps);
  };
  const bool vec = (width & 3) == 0 && ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) |
                                         reinterpret_cast<uintptr_t>(m) | reinterpret_cast<uintptr_t>(v)) & 15u) == 0;
  if (vec) {
    // rows of a multiple of four floats on 16-byte boundaries (quaternions, SH rows):
    // four elements of one row per thread and 16-byte accesses, one visibility test
    // per vector; the same per-element update
    const int w4 = width >> 2;
    const int64_t total4 = n * w4;
    float4 *p4 = reinterpret_cast<float4 *>(p), *m4 = reinterpret_cast<float4 *>(m), *v4 = reinterpret_cast<float4 *>(v);
    const float4 *g4 = reinterpret_cast<const float4 *>(g);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total4; i += stride) {
      if (radius && !visible(i / w4)) continue;
      const float4 gi = g4[i];
      float4 pi = p4[i], mi = m4[i], vi = v4[i];
      update(pi.x, mi.x, vi.x, gi.x);
      update(pi.y, mi.y, vi.y, gi.y);
      update(pi.z, mi.z, vi.z, gi.z);
      update(pi.w, mi.w, vi.w, gi.w);
      m4[i] = mi;
      v4[i] = vi;
      p4[i] = pi;
    }
    return;
  }
  const int64_t total = n * width;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += stride) {
    if (radius && !visible(i / width)) continue;
    float pi = p[i], mi = m[i], vi = v[i];
    update(pi, mi, vi, g[i]);
    m[i] = mi;
    v[i] = vi;
    p[i] = pi;
  }
}

// Bound by HBM. The grid is what the device keeps resident, and takes one group after the other:
// a grid of eight blocks per SM and group ran as one full round and a partial one
// (1.2M Gaussians, degree 3, 64% seen: 306 -> 274 us, 300k 91 -> 79; six blocks per SM and group
// 348 us, 64 of them 419, four resident instead of five 300). With few parameters each group
// has blocks of its own (gridDim.y): one group after the other is then five round trips to memory
// in turn (500 Gaussians, degree 3, 30% seen, 8.0 -> 5.1 us; 10k of degree 0 7.8 -> 5.4; at 10k of
// degree 3 one after the other 9.8 against 20).
__global__ void __launch_bounds__(256, 5) adam_kernel(gs_params_out_t P, gs_param_grads_t G, gs_adam_state_t S, int64_t n, int32_t sh_width,
                            float5_t step_size, float beta1, float beta2, float eps, float sqrt_bc2,
                            const int32_t *__restrict__ radius, int32_t n_views) {
#pragma unroll 1
  for (int grp = blockIdx.y; grp < 5; grp += gridDim.y)
    adam_group(grp, P, G, S, n, sh_width, step_size.v[grp], beta1, beta2, eps, sqrt_bc2, radius, n_views);
}

__global__ void opacity_reset_kernel(float *__restrict__ logits, float *__restrict__ m, float *__restrict__ v,
                                     int64_t n, float cap) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    logits[i] = fminf(logits[i], cap);
    if (m) m[i] = 0.f;
    if (v) v[i] = 0.f;
  }
}

}  // namespace gs

using namespace gs;

extern "C" size_t gs_photometric_workspace_size(const gs_frame_t *frame) {
  if (!frame || frame->n_views <= 0 || frame->n_pixels <= 0) return 0;
  return sizeof(float) * kPlanes * 3 * (size_t)frame->n_pixels + 2 * sizeof(double) * (size_t)frame->n_views + 256;
}

extern "C" gs_status_t gs_photometric_loss_grad(const gs_frame_t *frame, const float *image, const float *target,
                                                float lambda, float *d_image, float *loss_dev, void *ws,
                                                size_t ws_bytes, gs_stream_t stream) {
  if (!frame || !frame->cams_dev || frame->n_views <= 0 || !image || !target || !d_image || !loss_dev || !ws)
    return GS_ERR_INVALID_ARG;
  if (!(lambda >= 0.f && lambda <= 1.f) || ws_bytes < gs_photometric_workspace_size(frame) ||
      (reinterpret_cast<uintptr_t>(ws) & 15u) != 0)
    return GS_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  const int64_t stride = 3 * frame->n_pixels;
  // the FP64 sums first: the planes may hold an odd number of floats
  double *l1 = static_cast<double *>(ws), *ssim = l1 + frame->n_views;
  float *planes = reinterpret_cast<float *>(ssim + frame->n_views);
  GS_CUDA_TRY(cudaMemsetAsync(l1, 0, 2 * sizeof(double) * frame->n_views, s));
  const dim3 grid((frame->max_width + kTx - 1) / kTx, (frame->max_height + kTy - 1) / kTy, 3 * frame->n_views);
  GS_CUDA_TRY(cudaFuncSetAttribute(ssim_map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SsimTile)));
  GS_CUDA_TRY(cudaFuncSetAttribute(ssim_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradTile)));
  ssim_map_kernel<<<grid, kSsimThreads, sizeof(SsimTile), s>>>(frame->cams_dev, image, target, planes, stride, l1,
                                                               ssim);
  GS_LAUNCH_CHECK();
  ssim_grad_kernel<<<grid, kSsimThreads, sizeof(GradTile), s>>>(frame->cams_dev, image, target, planes, stride, lambda,
                                                                l1, ssim, loss_dev, d_image);
  GS_LAUNCH_CHECK();
  return GS_OK;
}

extern "C" gs_status_t gs_adam_step(const gs_adam_cfg_t *cfg, gs_params_out_t *params, int64_t n, int32_t sh_stride,
                                    const gs_param_grads_t *grads, gs_adam_state_t *state, const int32_t *radius,
                                    int32_t n_views, gs_stream_t stream) {
  if (!cfg || !params || !grads || !state || n < 0 || sh_stride < 1 || cfg->step < 1) return GS_ERR_INVALID_ARG;
  if (radius && n_views < 1) return GS_ERR_INVALID_ARG;
  if (!params->means || !params->log_scales || !params->quats || !params->opacity_logits || !params->sh ||
      !grads->d_means || !grads->d_log_scales || !grads->d_quats || !grads->d_opacity_logits || !grads->d_sh)
    return GS_ERR_INVALID_ARG;
  for (int k = 0; k < 5; ++k)
    if (!state->m[k] || !state->v[k]) return GS_ERR_INVALID_ARG;
  if (n == 0) return GS_OK;
  const double bc1 = 1.0 - std::pow(cfg->beta1, (double)cfg->step);
  const double bc2 = 1.0 - std::pow(cfg->beta2, (double)cfg->step);
  float5_t ss;
  for (int k = 0; k < 5; ++k) ss.v[k] = (float)(cfg->lr[k] / bc1);
  const int64_t widest = n * 3 * (int64_t)sh_stride;
  int per_sm = 0;
  GS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, adam_kernel, 256, 0));
  const int64_t blocks = (widest + 255) / 256;
  const bool few = blocks <= 2 * num_sms();   // five groups of them: two rounds at most
  const dim3 grid((unsigned)std::min<int64_t>(blocks, (int64_t)num_sms() * std::max(per_sm, 1)), few ? 5 : 1);
  adam_kernel<<<grid, 256, 0, as_stream(stream)>>>(*params, *grads, *state, n, 3 * sh_stride, ss, (float)cfg->beta1,
                                                 (float)cfg->beta2, cfg->eps, (float)std::sqrt(bc2), radius, n_views);
  GS_LAUNCH_CHECK();
  return GS_OK;
}

extern "C" gs_status_t gs_opacity_reset(float *opacity_logits, float *m, float *v, int64_t n, float max_opacity,
                                        gs_stream_t stream) {
  if (!opacity_logits || n < 0 || !(max_opacity > 0.f && max_opacity < 1.f)) return GS_ERR_INVALID_ARG;
  if (n == 0) return GS_OK;
  const float cap = (float)std::log((double)max_opacity / (1.0 - (double)max_opacity));
  const int grid = (int)std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8);
  opacity_reset_kernel<<<grid, 256, 0, as_stream(stream)>>>(opacity_logits, m, v, n, cap);
  GS_LAUNCH_CHECK();
  return GS_OK;
}
