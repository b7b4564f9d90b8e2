// Spatial SVGF denoiser (Schied et al. 2017 with its temporal parts removed,
// as the paper applies it to its raw Monte Carlo frames, Sec. 4.1; the depth
// gradient comes from the depth map offset by one pixel, supplementary
// "Rendering Details").  One thread per pixel:
//   svgf_variance_kernel: luminance variance from 7 x 7 depth/normal-weighted
//     moments (no history to estimate it from);
//   svgf_atrous_kernel:   one a-trous pass of the 5 x 5 B3 spline at step
//     2^i with depth, normal and variance-scaled luminance edge-stopping;
//     colour and variance travel together as float4 (rgb, Var).
// The image (16 B of colour, 4 B of depth and 16 B of normal per pixel) is a
// few MB at 800 x 800 and stays in L2 across the passes; taps hit L1.  The
// kernels are bound by instruction issue, so a tap is kept short:
//   - the edge-stopping functions multiply to one power of two, w = 2^-(a_z +
//     a_l + sigma_n L) in units of log2(e), L = -ln(n . n') (edge_weights below);
//   - the depth term's divisor depends on the offset alone and is equal for
//     opposite offsets: 12 (24 in the 7 x 7 window) reciprocals per pixel
//     instead of 25 (49) divisions;
//   - blocks whose whole window lies inside the image address taps by
//     constant offsets from one row pointer, without bounds tests;
//   - a window row's taps are loaded before any is weighted, and share one
//     test for the logarithm's series (270 us with a test per tap).
// 800 x 800, five passes: 229 us; with expf twice, powf and a division per
// tap 596 us (error against 64 bits 2.7e-7 both).
#include "device_common.cuh"

namespace rtk {
namespace {

constexpr float kEps = 1e-10f;
constexpr float kLog2e = 1.44269504088896340736f;
constexpr float kOutside = 1e30f;   // the exponent of a tap outside the image: weight 0
constexpr int kBX = 32, kBY = 8;

__device__ __forceinline__ float luminance(float4 c) { return 0.2126f * c.x + 0.7152f * c.y + 0.0722f * c.z; }

// forward differences of the depth map, backward at the last column / row
__device__ __forceinline__ float2 depth_gradient(const float* __restrict__ z, int W, int H, int x, int y) {
  const float zc = __ldg(z + y * W + x);
  float gx = 0.f, gy = 0.f;
  if (W > 1) gx = x + 1 < W ? __ldg(z + y * W + x + 1) - zc : zc - __ldg(z + y * W + x - 1);
  if (H > 1) gy = y + 1 < H ? __ldg(z + (y + 1) * W + x) - zc : zc - __ldg(z + (y - 1) * W + x);
  return make_float2(gx, gy);
}

// sigma_n in units of log2(e); the largest exponents stay finite (times L = 0 they have to give 0)
__device__ __forceinline__ float normal_exponent(float sigma_n) { return fminf(sigma_n * kLog2e, 3.402823466e38f); }

// -ln(c) for c = n . n' by the series of d = 1 - c (exact for c in [1/2, 2]), d + d^2/2 + ... + d^9/9.  For |d| < 1/8,
// which neighbouring taps of a smooth surface have, the remainder is below 2^-28 of the sum.
__device__ __forceinline__ float neg_ln_series(float d) {
  float s = 1.0f / 9.0f;
  s = fmaf(s, d, 1.0f / 8.0f);
  s = fmaf(s, d, 1.0f / 7.0f);
  s = fmaf(s, d, 1.0f / 6.0f);
  s = fmaf(s, d, 1.0f / 5.0f);
  s = fmaf(s, d, 1.0f / 4.0f);
  s = fmaf(s, d, 1.0f / 3.0f);
  s = fmaf(s, d, 0.5f);
  return fmaf(s * d, d, d);
}

// Normals that are not of unit length (averaged ones, say) scale all weights of a pixel alike, by about |n|^(2 sigma_n),
// which leaves the range of a float already for |n|^2 = 1/2.  Both filters form ratios of sums of equal degree in the
// weights, so the pixel's own normal is divided by |n|^2 where that power is far off 1: its own weight is 1 again.
template <bool NORMAL>
__device__ __forceinline__ f3 centre_normal(float4 n4, float sn) {
  const f3 n = xyz(n4);
  const float s = dot(n, n);
  return NORMAL && sn * fabsf(1.0f - s) > 16.0f ? n * __fdividef(1.0f, s) : n;
}

// Weights w_z w_n w_l of a row of D taps, each one power of two: a[k] is log2(e) times the depth and luminance exponent
// (>= 0), c[k] = n . n', sn = sigma_n log2(e); NORMAL: sigma_n > 0.  The row takes the series as a whole (one test per
// row and no divergence on smooth surfaces), or the library logarithm (a normal edge; c <= 0 or NaN: weight 0).
template <bool NORMAL, int D>
__device__ __forceinline__ void edge_weights(float (&a)[D], const float (&c)[D], float sn, float (&w)[D]) {
  if constexpr (NORMAL) {
    bool near = true;
#pragma unroll
    for (int k = 0; k < D; ++k) near = near && fabsf(1.0f - c[k]) < 0.125f;
    if (near) {
#pragma unroll
      for (int k = 0; k < D; ++k) a[k] = fmaf(sn, neg_ln_series(1.0f - c[k]), a[k]);
    } else {
#pragma unroll
      for (int k = 0; k < D; ++k) a[k] = fmaf(sn, -logf(fmaxf(c[k], 0.0f)), a[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < D; ++k) asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(w[k]) : "f"(-a[k]));   // max(0, c)^0 = 1
}

// The depth term's divisors as factors, log2(e) / (sigma_z |g . s| + eps), for the
// offsets of a (2R + 1)^2 window: entry (dy + R) * (2R + 1) + dx + R; opposite
// offsets share one, so only the window's first half is computed.  Both sides
// of the fast division are a quarter of that: it answers 0 for a divisor of
// 2^126 or more, which a background at the largest depths gives.
template <int R>
__device__ __forceinline__ void depth_divisors(float2 g, float step, float sigma_z, float (&inv)[(2 * R + 1) * (2 * R + 1)]) {
  constexpr int D = 2 * R + 1;
#pragma unroll
  for (int k = 0; k <= D * D / 2; ++k) {
    const float sx = step * (float)(k % D - R), sy = step * (float)(k / D - R);
    inv[k] = __fdividef(0.25f * kLog2e, fmaf(0.25f * sigma_z, fabsf(g.x * sx + g.y * sy), 0.25f * kEps));
    inv[D * D - 1 - k] = inv[k];
  }
}

template <bool INTERIOR, bool NORMAL>
__device__ __forceinline__ void variance_pixel(int W, int H, int x, int y, const float4* __restrict__ rad,
                                               const float* __restrict__ z, const float4* __restrict__ nrm,
                                               float sigma_z, float sigma_n, float4* __restrict__ out) {
  const int p = y * W + x;
  const float zp = __ldg(z + p);
  const float sn = normal_exponent(sigma_n);
  const f3 np_ = centre_normal<NORMAL>(__ldg(nrm + p), sn);
  float inv[49];
  depth_divisors<3>(depth_gradient(z, W, H, x, y), 1.0f, sigma_z, inv);
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll
  for (int dy = -3; dy <= 3; ++dy) {
    const int qy = y + dy;
    if (!INTERIOR && (qy < 0 || qy >= H)) continue;
    const int row = p + dy * W;
    float a[7], c[7], w[7], l[7];
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      const bool in = INTERIOR || (x + k - 3 >= 0 && x + k - 3 < W);
      a[k] = kOutside;
      c[k] = 1.0f;
      l[k] = 0.0f;
      if (in) {
        const int q = row + k - 3;
        a[k] = fabsf(zp - __ldg(z + q)) * inv[(dy + 3) * 7 + k];
        c[k] = dot(np_, xyz(__ldg(nrm + q)));
        l[k] = luminance(__ldg(rad + q));
      }
    }
    edge_weights<NORMAL>(a, c, sn, w);
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      s0 += w[k];
      s1 += w[k] * l[k];
      s2 += w[k] * l[k] * l[k];
    }
  }
  const float m1 = s1 / s0, m2 = s2 / s0;
  const float4 c = __ldg(rad + p);
  out[p] = make_float4(c.x, c.y, c.z, fmaxf(0.0f, m2 - m1 * m1));
}

template <bool NORMAL>
__global__ void __launch_bounds__(kBX* kBY, 3)
svgf_variance_kernel(int W, int H, const float4* __restrict__ rad, const float* __restrict__ z,
                     const float4* __restrict__ nrm, float sigma_z, float sigma_n, float4* __restrict__ out) {
  const int gx = (W + kBX - 1) / kBX;   // blocks in row order on one grid axis: no limit on the height
  const int x0 = (int)(blockIdx.x % gx) * kBX, y0 = (int)(blockIdx.x / gx) * kBY;
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  if (x0 >= 3 && y0 >= 3 && x0 + kBX + 3 <= W && y0 + kBY + 3 <= H)
    variance_pixel<true, NORMAL>(W, H, x, y, rad, z, nrm, sigma_z, sigma_n, out);
  else if (x < W && y < H)
    variance_pixel<false, NORMAL>(W, H, x, y, rad, z, nrm, sigma_z, sigma_n, out);
}

template <bool INTERIOR, bool NORMAL>
__device__ __forceinline__ void atrous_pixel(int W, int H, int step, int x, int y, const float4* __restrict__ in,
                                             const float* __restrict__ z, const float4* __restrict__ nrm,
                                             float sigma_z, float sigma_n, float sigma_l, float4* __restrict__ out) {
  const int p = y * W + x;
  // 3 x 3 Gaussian of the variance, out-of-image taps skipped
  float gs = 0.f, gw = 0.f;
#pragma unroll
  for (int dy = -1; dy <= 1; ++dy) {
    if (!INTERIOR && (y + dy < 0 || y + dy >= H)) continue;
#pragma unroll
    for (int dx = -1; dx <= 1; ++dx) {
      if (!INTERIOR && (x + dx < 0 || x + dx >= W)) continue;
      const float w = (dx == 0 ? 2.f : 1.f) * (dy == 0 ? 2.f : 1.f);
      gs += w * __ldg(&in[p + dy * W + dx].w);
      gw += w;
    }
  }
  const float inv_l = kLog2e / (sigma_l * sqrtf(fmaxf(gs / gw, 0.0f)) + kEps);
  const float4 cp = __ldg(in + p);
  const float lp = luminance(cp);
  const float zp = __ldg(z + p);
  const float sn = normal_exponent(sigma_n);
  const f3 np_ = centre_normal<NORMAL>(__ldg(nrm + p), sn);
  float inv[25];
  depth_divisors<2>(depth_gradient(z, W, H, x, y), (float)step, sigma_z, inv);
  constexpr float h1[5] = {1.f / 16.f, 1.f / 4.f, 3.f / 8.f, 1.f / 4.f, 1.f / 16.f};
  float ws = 0.f, ax = 0.f, ay = 0.f, az = 0.f, av = 0.f;
#pragma unroll
  for (int dy = -2; dy <= 2; ++dy) {
    const int qy = y + step * dy;
    if (!INTERIOR && (qy < 0 || qy >= H)) continue;
    const int row = p + step * dy * W;
    float4 cq[5];
    float a[5], c[5], w[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const int qx = x + step * (k - 2);
      const bool in_x = INTERIOR || (qx >= 0 && qx < W);
      a[k] = kOutside;
      c[k] = 1.0f;
      cq[k] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (in_x) {
        const int q = row + step * (k - 2);
        cq[k] = __ldg(in + q);
        a[k] = fmaf(fabsf(lp - luminance(cq[k])), inv_l, fabsf(zp - __ldg(z + q)) * inv[(dy + 2) * 5 + k]);
        c[k] = dot(np_, xyz(__ldg(nrm + q)));
      }
    }
    edge_weights<NORMAL>(a, c, sn, w);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      const float wk = h1[dy + 2] * h1[k] * w[k];
      ws += wk;
      ax += wk * cq[k].x;
      ay += wk * cq[k].y;
      az += wk * cq[k].z;
      av += wk * wk * cq[k].w;
    }
  }
  const float inv_w = 1.0f / ws;
  out[p] = make_float4(ax * inv_w, ay * inv_w, az * inv_w, av * inv_w * inv_w);
}

template <bool NORMAL>
__global__ void __launch_bounds__(kBX* kBY, 3)
svgf_atrous_kernel(int W, int H, int step, const float4* __restrict__ in, const float* __restrict__ z,
                   const float4* __restrict__ nrm, float sigma_z, float sigma_n, float sigma_l,
                   float4* __restrict__ out) {
  const int gx = (W + kBX - 1) / kBX;   // blocks in row order on one grid axis: no limit on the height
  const int x0 = (int)(blockIdx.x % gx) * kBX, y0 = (int)(blockIdx.x / gx) * kBY;
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const int m = 2 * step;   // the window's reach
  if (x0 >= m && y0 >= m && x0 + kBX + m <= W && y0 + kBY + m <= H)
    atrous_pixel<true, NORMAL>(W, H, step, x, y, in, z, nrm, sigma_z, sigma_n, sigma_l, out);
  else if (x < W && y < H)
    atrous_pixel<false, NORMAL>(W, H, step, x, y, in, z, nrm, sigma_z, sigma_n, sigma_l, out);
}

template <bool NORMAL>
cudaError_t run_denoise(int W, int H, const float4* rad, const float* z, const float4* nrm, int iterations,
                        float sigma_z, float sigma_n, float sigma_l, float4* a, float4* b, cudaStream_t s) {
  const dim3 block(kBX, kBY);
  const unsigned grid = (unsigned)((W + kBX - 1) / kBX) * (unsigned)((H + kBY - 1) / kBY);
  svgf_variance_kernel<NORMAL><<<grid, block, 0, s>>>(W, H, rad, z, nrm, sigma_z, sigma_n, a);
  cudaError_t e = cudaGetLastError();
  for (int i = 0; i < iterations && e == cudaSuccess; ++i) {
    svgf_atrous_kernel<NORMAL><<<grid, block, 0, s>>>(W, H, 1 << i, a, z, nrm, sigma_z, sigma_n, sigma_l, b);
    e = cudaGetLastError();
    float4* t = a;
    a = b;
    b = t;
  }
  return e;
}

}  // namespace

cudaError_t launch_denoise(int W, int H, const float4* rad, const float* z, const float4* nrm, int iterations,
                           float sigma_z, float sigma_n, float sigma_l, float4* work, float4* out, cudaStream_t s) {
  // the last pass writes `out`: start in `out` for an even pass count, in `work` for an odd one
  float4* a = (iterations % 2 == 0) ? out : work;
  float4* b = (iterations % 2 == 0) ? work : out;
  return sigma_n > 0.0f ? run_denoise<true>(W, H, rad, z, nrm, iterations, sigma_z, sigma_n, sigma_l, a, b, s)
                                 : run_denoise<false>(W, H, rad, z, nrm, iterations, sigma_z, sigma_n, sigma_l, a, b, s);
}

}  // namespace rtk
