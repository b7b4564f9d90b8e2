// rt_set_params' device work in one launch: the FP32 and BF16 weight images,
// and the texel distribution of the bound environment map.  They are
// independent (the BF16 image is formed from the blobs, not from the FP32
// image), so the rows of the map and both images share a grid, and the CTA
// that finishes the last row builds the marginal; as four dependent launches
// they took 19 us for a 256 x 512 map, most of it launch latency and drain;
// together 10.9 us.
//
// Texel distribution for the light strategy of the MIS primary sampler (Sec. 4.1): luminance 0.2126 R + 0.7152 G +
// 0.0722 B, negative parts clipped, plus 1e-6; conditional CDFs along each
// row and a marginal CDF over rows.  The inversion of these CDFs decides
// integers, so they are built in float32 with every product and sum
// rounded on its own (no contraction), running sums in index order, one
// correctly rounded division by the total, and the last entry set to 1.
// Cutpoint tables over each CDF then start the sampler's bisection close to
// its answer.
//
// The running sums bound this set-up: float32 additions in index order are one
// dependent chain, 4 cycles per texel, and nothing may reorder them.  So only
// the chain is serial: a CTA per row loads the row's texels coalesced and forms
// their luminances in shared memory, one thread runs the chain over it 16
// texels at a time (the next 16 are read while these are added), and all
// threads divide, write the row and answer its cutpoints from shared memory.
// With the chain in global memory (one thread per row, a dependent load and a
// strided store per texel) a 256 x 512 map took 403 us and its marginal 34 us.
#include "mis.cuh"
#include "repack.cuh"

namespace rtk {
namespace {

constexpr int kCdfThreads = 128;
constexpr int kPackBlocks = (WPACK_FLOATS + kCdfThreads - 1) / kCdfThreads;
constexpr int kBf16Blocks = (WBF16_BYTES / 2 + kCdfThreads - 1) / kCdfThreads;

// v[0..n) -> its running sums, in index order, each rounded to float32; the last one is the total.
__device__ __forceinline__ void running_sum(float* v, int n) {
  float s = 0.0f;
  float4* v4 = reinterpret_cast<float4*>(v);
  const int blocks = n / 16;
  float4 a[4];
  if (blocks > 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = v4[k];
  for (int b = 0; b < blocks; ++b) {
    float4 nx[4];
    const int nb = min(b + 1, blocks - 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) nx[k] = v4[4 * nb + k];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k].x = s = __fadd_rn(s, a[k].x);
      a[k].y = s = __fadd_rn(s, a[k].y);
      a[k].z = s = __fadd_rn(s, a[k].z);
      a[k].w = s = __fadd_rn(s, a[k].w);
      v4[4 * b + k] = a[k];
      a[k] = nx[k];
    }
  }
  for (int c = 16 * blocks; c < n; ++c) v[c] = s = __fadd_rn(s, v[c]);
}

// Turn the running sums v[0..n) into the CDF cdf[0..n] (0 first, 1 last) and answer its cutpoint table:
// entry j is the bisection's answer for u = j / 2^shift (exact in float32).
__device__ __forceinline__ void finish_cdf(float* v, int n, float* __restrict__ cdf, int* __restrict__ guide,
                                           int shift) {
  const float total = v[n - 1];
  __syncthreads();   // every thread has read the total
  for (int c = threadIdx.x; c < n; c += kCdfThreads) {
    const float q = c + 1 < n ? __fdiv_rn(v[c], total) : 1.0f;
    v[c] = q;
    cdf[c + 1] = q;
  }
  if (threadIdx.x == 0) cdf[0] = 0.0f;
  __syncthreads();
  const int G = 1 << shift;
  for (int j = threadIdx.x; j < G; j += kCdfThreads) {
    const float u = (float)j * (1.0f / (float)G);
    int lo = 0, hi = n;   // bisection with cdf[k] = v[k - 1] for k >= 1
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (v[mid - 1] <= u) lo = mid;
      else hi = mid;
    }
    guide[j] = lo;
  }
}

// CTA r < H: the conditional CDF of row r, its cutpoints, and the row's total into cdf_m[r + 1]; the CTA that finishes
// last (the H-th count of *done, zero before the launch) turns the totals into the marginal CDF and answers its cutpoints.
// *done_next, the next call's count, is cleared here: no count outlives one call.
// Further CTAs: kCdfThreads elements of the FP32 image each, then of the BF16 image.
__global__ void __launch_bounds__(kCdfThreads)
set_params_kernel(const float* __restrict__ bw, const float* __restrict__ iw, int lf, float* __restrict__ wpack,
                  uint8_t* __restrict__ wbf16, const float4* __restrict__ env, int H, int W, float* cdf_m,
                  float* __restrict__ cdf_c, int* __restrict__ guide_m, int gm_shift, int* __restrict__ guide_c,
                  int gc_shift, uint32_t* done, uint32_t* done_next) {
  extern __shared__ float4 cdf_smem4[];
  float* v = reinterpret_cast<float*>(cdf_smem4);
  const int r = blockIdx.x;
  if (r >= H) {
    int e = (r - H) * kCdfThreads + threadIdx.x;
    if (e < kPackBlocks * kCdfThreads) {
      if (e < WPACK_FLOATS) wpack[e] = packed_value(bw, iw, lf, e);
      return;
    }
    e -= kPackBlocks * kCdfThreads;
    if (e < WBF16_BYTES / 2)
      reinterpret_cast<__nv_bfloat16*>(wbf16)[e] =
          bf16_image_value(2 * e, [&](int k) { return packed_value(bw, iw, lf, k); });
    return;
  }
  for (int c = threadIdx.x; c < W; c += kCdfThreads) {
    const float4 e = env[(size_t)r * W + c];
    const float lum = __fadd_rn(__fadd_rn(__fmul_rn(e.x, 0.2126f), __fmul_rn(e.y, 0.7152f)), __fmul_rn(e.z, 0.0722f));
    v[c] = __fadd_rn(fmaxf(lum, 0.0f), 1e-6f);
  }
  __syncthreads();
  __shared__ uint32_t last;
  if (threadIdx.x == 0) {
    running_sum(v, W);
    __stcg(cdf_m + r + 1, v[W - 1]);   // turned into the marginal CDF by the last CTA
    __threadfence();
    last = atomicAdd(done, 1u) + 1u == (uint32_t)H;
    if (r == 0) *done_next = 0u;
  }
  __syncthreads();
  finish_cdf(v, W, cdf_c + (size_t)r * (W + 1), guide_c + ((size_t)r << gc_shift), gc_shift);
  if (!last) return;
  __threadfence();   // the other rows' totals are visible
  __syncthreads();   // v is read
  for (int k = threadIdx.x; k < H; k += kCdfThreads) v[k] = __ldcg(cdf_m + k + 1);
  __syncthreads();
  if (threadIdx.x == 0) running_sum(v, H);
  __syncthreads();
  finish_cdf(v, H, cdf_m, guide_m, gm_shift);
}

}  // namespace

cudaError_t launch_set_params(const float* brdf_w, const float* irt_w, int lf, float* wpack, uint8_t* wbf16,
                              const float4* env, int H, int W, float* cdf_m, float* cdf_c, int* guide_m, int gm_shift,
                              int* guide_c, int gc_shift, uint32_t* done, uint32_t* done_next, cudaStream_t s) {
  // a row or column of at most 8192 floats fits the 48 KB of shared memory that need no opt-in
  const size_t smem = ((size_t)(H > W ? H : W) + 3) / 4 * 16;
  set_params_kernel<<<H + kPackBlocks + kBf16Blocks, kCdfThreads, smem, s>>>(
      brdf_w, irt_w, lf, wpack, wbf16, env, H, W, cdf_m, cdf_c, guide_m, gm_shift, guide_c, gc_shift, done, done_next);
  return cudaGetLastError();
}

}  // namespace rtk
