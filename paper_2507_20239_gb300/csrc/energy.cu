// Energy of training images across resolutions, for the coarse-to-fine schedule
// (Sec. "Energy-aware multi-resolution"): the anti-aliased bilinear downscale
// D_r and the L1 norm of the 2D Fourier magnitude, ||E(I)||_1.
//
// D_r: separable triangle filter whose support widens with the scale s = W / W_r
// (W_r = floor(W/r + 1/2)); output column j samples the input at c = (j + 1/2) s - 1/2
// with weights max(0, 1 - |k - c| / s) over the input columns k inside the image,
// normalised to sum 1; rows likewise.
//
// ||E(I)||_1: a 2D DFT of each channel as two 1D DFT passes -- rows (real input) and
// columns (complex input, the magnitudes to about 2^-46 in FP32 pairs, summed as such per
// warp and added once per warp in FP64), each a direct sum with twiddles from a shared table indexed by n k mod N, the
// index advanced incrementally; no FFT library is used. The direct sum keeps every
// coefficient's FP32 rounding sequence independent of how N factors.
#include <algorithm>

#include "gs_common.cuh"

namespace gs {

constexpr int kEnergyMaxDim = 4096;

__device__ __forceinline__ void aa_taps(int j, int n_in, int n_out, float &c, float &s, int &k0, int &k1,
                                        float &norm) {
  s = (float)n_in / (float)n_out;
  c = ((float)j + 0.5f) * s - 0.5f;
  k0 = max(0, (int)ceilf(c - s));
  k1 = min(n_in - 1, (int)floorf(c + s));
  float sum = 0.f;
  for (int k = k0; k <= k1; ++k) sum += fmaxf(0.f, 1.f - fabsf((float)k - c) / s);
  norm = 1.f / sum;
}

// Any factor: every weight evaluated where it is used.
__global__ void downscale_kernel(const float *__restrict__ img, int C, int H, int W, float *__restrict__ out,
                                 int Hr, int Wr) {
  const int64_t total = (int64_t)Hr * Wr;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < total; p += (int64_t)gridDim.x * blockDim.x) {
    const int y = (int)(p / Wr), x = (int)(p - (int64_t)y * Wr);
    float cx, sx, nx, cy, sy, ny;
    int x0, x1, y0, y1;
    aa_taps(x, W, Wr, cx, sx, x0, x1, nx);
    aa_taps(y, H, Hr, cy, sy, y0, y1, ny);
    for (int ch = 0; ch < C; ++ch) {
      const float *src = img + (int64_t)ch * H * W;
      float acc = 0.f;
      for (int ky = y0; ky <= y1; ++ky) {
        const float wy = fmaxf(0.f, 1.f - fabsf((float)ky - cy) / sy);
        float row = 0.f;
        for (int kx = x0; kx <= x1; ++kx) row = fmaf(fmaxf(0.f, 1.f - fabsf((float)kx - cx) / sx), src[(int64_t)ky * W + kx], row);
        acc = fmaf(wy, row, acc);
      }
      out[(int64_t)ch * Hr * Wr + p] = acc * nx * ny;
    }
  }
}

// Factors whose filters have at most kMaxTaps taps (r <= 16: the schedule's are up to 8):
// a block's 32 x 8 output pixels share 32 column and 8 row filters, evaluated once into
// shared memory (one division per weight instead of one per tap, pixel and channel, which
// is what the general kernel spends its time on). blockIdx.z is the channel. Same sums in
// the same order, so the same bits: scales 2, 3, 4 of a 3 x 826 x 1246
// image 73 -> 38 us.
constexpr int kMaxTaps = 36, kDsX = 32, kDsY = 8;

__global__ void __launch_bounds__(kDsX *kDsY) downscale_taps_kernel(const float *__restrict__ img, int H, int W,
                                                                    float *__restrict__ out, int Hr, int Wr) {
  __shared__ float s_wx[kMaxTaps][kDsX], s_wy[kMaxTaps][kDsY];
  __shared__ float s_nx[kDsX], s_ny[kDsY];
  __shared__ int s_x0[kDsX], s_x1[kDsX], s_y0[kDsY], s_y1[kDsY];
  const int t = threadIdx.y * kDsX + threadIdx.x;
  if (t < kDsX + kDsY) {
    const bool col = t < kDsX;
    const int i = col ? t : t - kDsX;
    const int j = (col ? blockIdx.x * kDsX : blockIdx.y * kDsY) + i;
    float c = 0.f, sc = 1.f, norm = 0.f;
    int k0 = 0, k1 = -1;
    if (j < (col ? Wr : Hr)) aa_taps(j, col ? W : H, col ? Wr : Hr, c, sc, k0, k1, norm);
    for (int k = k0; k <= k1; ++k) {
      const float w = fmaxf(0.f, 1.f - fabsf((float)k - c) / sc);
      if (col) s_wx[k - k0][i] = w; else s_wy[k - k0][i] = w;
    }
    if (col) {
      s_x0[i] = k0; s_x1[i] = k1; s_nx[i] = norm;
    } else {
      s_y0[i] = k0; s_y1[i] = k1; s_ny[i] = norm;
    }
  }
  __syncthreads();
  const int x = blockIdx.x * kDsX + threadIdx.x, y = blockIdx.y * kDsY + threadIdx.y;
  if (x >= Wr || y >= Hr) return;
  const int x0 = s_x0[threadIdx.x], x1 = s_x1[threadIdx.x], y0 = s_y0[threadIdx.y], y1 = s_y1[threadIdx.y];
  const float *src = img + (int64_t)blockIdx.z * H * W;
  float acc = 0.f;
  for (int ky = y0; ky <= y1; ++ky) {
    const float *line = src + (int64_t)ky * W + x0;
    float row = 0.f;
    for (int k = 0; k <= x1 - x0; ++k) row = fmaf(s_wx[k][threadIdx.x], line[k], row);
    acc = fmaf(s_wy[ky - y0][threadIdx.y], row, acc);
  }
  out[(int64_t)blockIdx.z * Hr * Wr + (int64_t)y * Wr + x] = acc * s_nx[threadIdx.x] * s_ny[threadIdx.y];
}

// tw[q] = exp(-2 pi i q / N), q in [0, N), of the rows (N = W) and of the columns (N = H),
// computed once per call: the double-precision sines, done by every block of a DFT pass,
// cost more than the pass (FP64 runs at 1/64 of the FP32 rate here). Blocks of one warp: the FP64
// pipes of many SMs instead of one. Clears the sum as well (a launch less; the two together 64 x 64
// 16.3 -> 12.8 us for the call, 3 x 623 x 413 90.6 -> 87.8).
constexpr int kTwThreads = 32;

__global__ void __launch_bounds__(kTwThreads) twiddles_kernel(float2 *__restrict__ tw_w, int W,
                                                              float2 *__restrict__ tw_h, int H, double *sum) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *sum = 0.0;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= W + H) return;
  const int N = i < W ? W : H, q = i < W ? i : i - W;
  double sn, cs;
  sincospi(2.0 * (double)q / (double)N, &sn, &cs);
  (i < W ? tw_w : tw_h)[q] = make_float2((float)cs, (float)-sn);
}

// Twiddle q sits at slot q + q / 16 of the shared table: lanes of consecutive k read
// q = n k mod N at stride n, which without the padding puts 2 to 16 lanes on one bank
// for every even n.
__device__ __forceinline__ int tw_slot(int q) { return q + (q >> 4); }
static int tw_slots(int N) { return N + (N >> 4) + 1; }

__device__ __forceinline__ void load_twiddles(float2 *s_tw, const float2 *__restrict__ tw, int N) {
  for (int q = threadIdx.x; q < N; q += blockDim.x) s_tw[tw_slot(q)] = tw[q];
}

// Both passes are a direct O(N^2) sum per coefficient, in the order n = 0, 1, ..., on the
// FP32 pipes. A thread keeps 8 or 16 lines (rows, or columns) of one or two (KK) frequencies in
// registers, so a twiddle serves all of its lines and a line's value its frequencies; neighbouring
// lines are packed pairs (f32x2: the same operations and roundings at half the issue slots).
// With one line and one frequency per thread the passes ran at the rate of their
// shared-memory loads (a conflicted twiddle per two FMAs).
// The input is real, so X[h][W - k] = conj X[h][k] and column W - k has the magnitudes of
// column k: only k = 0 .. W / 2 are computed, the others counted with weight 2.
// 3 x 826 x 1246: row pass ~1770 -> 216 us unpacked, 187 packed; column pass ~1390 -> 247 and 237
// (229 us of FMAs in the two at the FP32 peak), pairs of (re, im) instead of two columns, which
// need every value twice, 274; 3 x 207 x 312: 30 -> 14 and 21 -> 14. The coefficients have the same bits.
constexpr int kDftThreads = 64;
constexpr int kDftCols = 8;                     // columns per thread (column pass)
constexpr int kDftChunk = 64;                   // line positions staged at a time

// X[line][k] = sum_n I[line][n] exp(-2 pi i n k / W), line = channel * H + row.
template <int ROWS, int KK>
__global__ void __launch_bounds__(kDftThreads, ROWS * KK > 16 ? 6 : 12) dft_rows_kernel(
    const float *__restrict__ img, int64_t lines, int W, int K, const float2 *__restrict__ tw, float2 *__restrict__ X) {
  constexpr int kPad = ROWS + 4;   // staged position: 16-byte aligned, 4-way at most when filled
  extern __shared__ float4 s_raw[];
  float *s_x = reinterpret_cast<float *>(s_raw);                               // [kDftChunk][kPad]
  float2 *s_tw = reinterpret_cast<float2 *>(s_x + kDftChunk * kPad);
  const int64_t l0 = (int64_t)blockIdx.x * ROWS;
  load_twiddles(s_tw, tw, W);
  int k[KK], q[KK];
  float2 re[KK][ROWS / 2], im[KK][ROWS / 2];
#pragma unroll
  for (int j = 0; j < KK; ++j) {
    const int kk = (blockIdx.y * KK + j) * kDftThreads + threadIdx.x;
    k[j] = kk < K ? kk : 0;
    q[j] = 0;
#pragma unroll
    for (int r = 0; r < ROWS / 2; ++r) re[j][r] = im[j][r] = make_float2(0.f, 0.f);
  }
  for (int n0 = 0; n0 < W; n0 += kDftChunk) {
    const int cnt = min(kDftChunk, W - n0);
    __syncthreads();
    for (int i = threadIdx.x; i < kDftChunk * ROWS; i += kDftThreads) {
      const int r = i / kDftChunk, n = i - r * kDftChunk;
      s_x[n * kPad + r] = n < cnt && l0 + r < lines ? img[(l0 + r) * W + n0 + n] : 0.f;
    }
    __syncthreads();
#pragma unroll 4
    for (int n = 0; n < cnt; ++n) {
      float2 x[ROWS / 2];
#pragma unroll
      for (int r = 0; r < ROWS / 2; r += 2) {
        const float4 v = *reinterpret_cast<const float4 *>(s_x + n * kPad + 2 * r);
        x[r] = make_float2(v.x, v.y);
        x[r + 1] = make_float2(v.z, v.w);
      }
#pragma unroll
      for (int j = 0; j < KK; ++j) {
        const float2 t = s_tw[tw_slot(q[j])];
#pragma unroll
        for (int r = 0; r < ROWS / 2; ++r) {
          re[j][r] = f2_fma(x[r], f2(t.x), re[j][r]);
          im[j][r] = f2_fma(x[r], f2(t.y), im[j][r]);
        }
        q[j] += k[j];
        q[j] = (int)min((uint32_t)q[j], (uint32_t)(q[j] - W));   // q mod W (q < 2 W)
      }
    }
  }
#pragma unroll
  for (int j = 0; j < KK; ++j) {
    const int kk = (blockIdx.y * KK + j) * kDftThreads + threadIdx.x;
    if (kk >= K) continue;
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
      if (l0 + r < lines)
        X[(l0 + r) * K + kk] = r & 1 ? make_float2(re[j][r / 2].y, im[j][r / 2].y)
                                     : make_float2(re[j][r / 2].x, im[j][r / 2].x);
  }
}

// (s, c) += weight |z|, |z| to about 2^-46 in FP32 pairs (the FP64 square root ran for
// longer than the DFT): z's squares as hi + lo exactly but for lo's last bits, m ~ sqrt(hi)
// and its correction (hi + lo - m^2) / (2 m), one rounding per operation as written (a
// contracted product would count its own rounding error twice). Outside the range where no term of
// that under- or overflows, the FP64 root, into `wide`. weight: 1 or 2.
__device__ __forceinline__ void add_magnitude(float re, float im, float weight, float &s, float &c, double &wide) {
  const float a = fmaxf(fabsf(re), fabsf(im)), b = fminf(fabsf(re), fabsf(im));
  if (!(a >= 1e-12f && fabsf(re) <= 1e15f && fabsf(im) <= 1e15f)) {
    if (re != 0.f || im != 0.f) wide += (double)weight * sqrt((double)re * re + (double)im * im);
    return;
  }
  const float a2 = __fmul_rn(a, a), b2 = __fmul_rn(b, b);
  const float hi = __fadd_rn(a2, b2);
  const float lo = __fadd_rn(__fsub_rn(b2, __fsub_rn(hi, a2)), __fadd_rn(__fmaf_rn(a, a, -a2), __fmaf_rn(b, b, -b2)));
  const float m = __fsqrt_rn(hi);
  const float e = __fmul_rn(__fadd_rn(__fmaf_rn(-m, m, hi), lo), __fdiv_rn(0.5f, m));
  pair_add(s, c, __fmul_rn(weight, m));
  c = __fadd_rn(c, __fmul_rn(weight, e));
}

// Y[m] = sum_h X[h][k] exp(-2 pi i h m / H) of kDftCols adjacent columns k (of the K kept)
// of one channel; adds sum |Y[m]| to *sum, columns that stand for W - k too twice.
template <int KK>
__global__ void __launch_bounds__(kDftThreads, KK > 1 ? 8 : 12) dft_cols_l1_kernel(
    const float2 *__restrict__ X, int H, int W, int K, const float2 *__restrict__ tw, double *sum) {
  extern __shared__ float4 s_raw[];
  float4 *s_x = s_raw;                          // [kDftChunk][kDftCols / 2]: (re, re, im, im) of two columns
  float2 *s_tw = reinterpret_cast<float2 *>(s_x + kDftChunk * kDftCols / 2);
  const int col_blocks = (K + kDftCols - 1) / kDftCols;
  const int ch = blockIdx.x / col_blocks, c0 = (blockIdx.x - ch * col_blocks) * kDftCols;
  const float2 *src = X + (int64_t)ch * H * K;
  load_twiddles(s_tw, tw, H);
  int m[KK], q[KK];
  float2 re[KK][kDftCols / 2], im[KK][kDftCols / 2];
#pragma unroll
  for (int j = 0; j < KK; ++j) {
    const int mm = (blockIdx.y * KK + j) * kDftThreads + threadIdx.x;
    m[j] = mm < H ? mm : 0;
    q[j] = 0;
#pragma unroll
    for (int c = 0; c < kDftCols / 2; ++c) re[j][c] = im[j][c] = f2(0.f);
  }
  for (int h0 = 0; h0 < H; h0 += kDftChunk) {
    const int cnt = min(kDftChunk, H - h0);
    __syncthreads();
    for (int i = threadIdx.x; i < kDftChunk * kDftCols; i += kDftThreads) {
      const int h = i / kDftCols, c = i - h * kDftCols;
      const float2 x = h < cnt && c0 + c < K ? src[(int64_t)(h0 + h) * K + c0 + c] : make_float2(0.f, 0.f);
      float *to = reinterpret_cast<float *>(s_x + i / 2) + (c & 1);
      to[0] = x.x;
      to[2] = x.y;
    }
    __syncthreads();
#pragma unroll 4
    for (int h = 0; h < cnt; ++h) {
      float4 x[kDftCols / 2];
#pragma unroll
      for (int c = 0; c < kDftCols / 2; ++c) x[c] = s_x[h * (kDftCols / 2) + c];
#pragma unroll
      for (int j = 0; j < KK; ++j) {
        const float2 t = s_tw[tw_slot(q[j])];
        const float2 tx = f2(t.x), ty = f2(t.y), ny = f2(-t.y);
#pragma unroll
        for (int c = 0; c < kDftCols / 2; ++c) {
          const float2 xr = f2(x[c].x, x[c].y), xi = f2(x[c].z, x[c].w);
          re[j][c] = f2_fma(xr, tx, f2_fma(xi, ny, re[j][c]));
          im[j][c] = f2_fma(xr, ty, f2_fma(xi, tx, im[j][c]));
        }
        q[j] += m[j];
        q[j] = (int)min((uint32_t)q[j], (uint32_t)(q[j] - H));
      }
    }
  }
  float part = 0.f, part_c = 0.f;
  double wide = 0.0;
#pragma unroll
  for (int j = 0; j < KK; ++j) {
    if ((blockIdx.y * KK + j) * kDftThreads + threadIdx.x >= H) continue;
#pragma unroll
    for (int c = 0; c < kDftCols; ++c) {
      const int k = c0 + c;
      const float2 r = re[j][c / 2], i = im[j][c / 2];
      if (k < K)
        add_magnitude(c & 1 ? r.y : r.x, c & 1 ? i.y : i.x, k == 0 || 2 * k == W ? 1.f : 2.f, part, part_c, wide);
    }
  }
  if (wide != 0.0) atomicAdd(sum, wide);
  warp_pair_sum(part, part_c);
  if ((threadIdx.x & 31) == 0) atomicAdd(sum, (double)part + (double)part_c);
}

static bool dims_ok(int C, int H, int W) {
  return C > 0 && H > 0 && W > 0 && H <= kEnergyMaxDim && W <= kEnergyMaxDim;
}

}  // namespace gs

using namespace gs;

extern "C" int32_t gs_downscaled_size(int32_t n, int32_t r) {
  if (n <= 0 || r < 1) return 0;
  const int64_t m = (2 * (int64_t)n + r) / (2 * (int64_t)r);   // floor(n / r + 1/2)
  return (int32_t)(m > 0 ? m : 1);
}

extern "C" gs_status_t gs_downscale(const float *image, int32_t C, int32_t H, int32_t W, int32_t r, float *out,
                                    gs_stream_t stream) {
  if (!image || !out || C <= 0 || H <= 0 || W <= 0 || r < 1) return GS_ERR_INVALID_ARG;
  const int Hr = gs_downscaled_size(H, r), Wr = gs_downscaled_size(W, r);
  // taps per axis: at most 2 s + 1 with s = W / Wr <= 1.5 r (Wr rounds W / r down to half), and
  // one more by the FP32 rounding of the positions up to 2^22 columns or rows; beyond, any number
  int64_t taps = kMaxTaps + 1;
  if (W <= 1 << 22 && H <= 1 << 22) taps = 2 * (int64_t)std::max((W + Wr - 1) / Wr, (H + Hr - 1) / Hr) + 2;
  const dim3 blocks((Wr + kDsX - 1) / kDsX, (Hr + kDsY - 1) / kDsY, C);
  // Steps of whole 32-byte sectors put 8 or 16 lanes of a load on one bank. On large images that is what both
  // kernels take their time from, and the general one, whose blocks read along one row, takes less of it:
  // tabulated and general, us, scale 8, 1 channel 4096 x 4096 94 / 84, 6000 x 4000 112 / 96, 3 channels 4096 x 3000
  // 166 / 138, 6000 x 4000 299 / 273; 3200 x 2400 46 / 43 and 116 / 116, 2600 x 2000 36 / 34 and 87 / 92; scale 16, 3
  // channels 4096 x 4096 422 / 392, 6000 x 4000 771 / 586. Other scales take the tables at any size.
  const bool conflicts = r % 8 == 0 && (int64_t)H * W >= 7000000;
  if (taps <= kMaxTaps && !conflicts && blocks.y <= 65535 && blocks.z <= 65535) {
    downscale_taps_kernel<<<blocks, dim3(kDsX, kDsY), 0, as_stream(stream)>>>(image, H, W, out, Hr, Wr);
  } else {
    const int64_t total = (int64_t)Hr * Wr;
    const int grid = (int)std::min<int64_t>((total + 255) / 256, (int64_t)num_sms() * 16);
    downscale_kernel<<<grid, 256, 0, as_stream(stream)>>>(image, C, H, W, out, Hr, Wr);
  }
  GS_LAUNCH_CHECK();
  return GS_OK;
}

extern "C" size_t gs_spectrum_workspace_size(int32_t C, int32_t H, int32_t W) {
  if (!dims_ok(C, H, W)) return 0;
  // the kept coefficients of the row pass, then both passes' twiddles
  return sizeof(float2) * ((size_t)C * H * (W / 2 + 1) + W + H);
}

extern "C" gs_status_t gs_spectrum_l1(const float *image, int32_t C, int32_t H, int32_t W, double *d_sum, void *ws,
                                      size_t ws_bytes, gs_stream_t stream) {
  if (!image || !d_sum || !ws || !dims_ok(C, H, W)) return GS_ERR_INVALID_ARG;
  if (ws_bytes < gs_spectrum_workspace_size(C, H, W) || (reinterpret_cast<uintptr_t>(ws) & 15u) != 0)
    return GS_ERR_INVALID_ARG;
  cudaStream_t s = as_stream(stream);
  const int K = W / 2 + 1;
  const int64_t lines = (int64_t)C * H;
  const int64_t col_blocks = (int64_t)C * ((K + kDftCols - 1) / kDftCols);
  const int64_t row_blocks = (lines + 15) / 16;   // of 16 lines
  if (row_blocks > 0x7fffffffll || col_blocks > 0x7fffffffll) return GS_ERR_INVALID_ARG;
  float2 *X = static_cast<float2 *>(ws);
  float2 *tw_w = X + lines * K, *tw_h = tw_w + W;
  twiddles_kernel<<<(W + H + kTwThreads - 1) / kTwThreads, kTwThreads, 0, s>>>(tw_w, W, tw_h, H, d_sum);
  GS_LAUNCH_CHECK();
  auto rows = [&](auto kernel, int per, int freqs) {
    const dim3 grid((unsigned)((lines + per - 1) / per), (K + kDftThreads * freqs - 1) / (kDftThreads * freqs));
    const size_t smem = sizeof(float) * kDftChunk * (per + 4) + sizeof(float2) * tw_slots(W);
    kernel<<<grid, kDftThreads, smem, s>>>(image, lines, W, K, tw_w, X);
  };
  auto cols = [&](auto kernel, int freqs) {
    const dim3 grid((unsigned)col_blocks, (H + kDftThreads * freqs - 1) / (kDftThreads * freqs));
    const size_t smem = sizeof(float2) * kDftChunk * kDftCols + sizeof(float2) * tw_slots(H);
    static_assert(sizeof(float2) * (kDftChunk * kDftCols + kEnergyMaxDim + kEnergyMaxDim / 16 + 1) <= 48 * 1024,
                  "fits the default shared-memory limit");
    kernel<<<grid, kDftThreads, smem, s>>>(X, H, W, K, tw_h, d_sum);
  };
  // The larger tiles reuse more per load, the smaller ones keep more warps at work, and on
  // images of few blocks, whose threads wait for one sum after another, that counts for more. Larger
  // and smaller, us: rows, at 9.2, 5.1, 3.0, 1.5, 0.8, 0.5 blocks of 16 x 128 per SM, 378 / 569,
  // 187 / 277, 95 / 114, 43 / 44, 35 / 29, 23 / 14; columns, at 10.8, 5.6, 5.0, 3.1, 1.5, 0.8 blocks of
  // 8 x 128, 237 / 259, 97 / 109, 84 / 85, 48 / 40, 24 / 20, 19 / 14.
  if (row_blocks * ((K + 2 * kDftThreads - 1) / (2 * kDftThreads)) >= num_sms())
    rows(dft_rows_kernel<16, 2>, 16, 2);
  else
    rows(dft_rows_kernel<8, 1>, 8, 1);
  GS_LAUNCH_CHECK();
  if (col_blocks * ((H + 2 * kDftThreads - 1) / (2 * kDftThreads)) >= 4 * num_sms())
    cols(dft_cols_l1_kernel<2>, 2);
  else
    cols(dft_cols_l1_kernel<1>, 1);
  GS_LAUNCH_CHECK();
  return GS_OK;
}
