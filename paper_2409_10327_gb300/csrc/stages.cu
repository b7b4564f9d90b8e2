// Stand-alone stage kernels: weight repacking, stage (a) encode, the direction
// sampler and stage (e) shading at one level, one thread per output item
// (stages (b) and (c), the MLPs, are in stages_mlp.cu).  They compute exactly
// what the fused kernel computes per sample and give each stage its own parity
// check.
#include "device_common.cuh"
#include "repack.cuh"

namespace rtk {

// ---- weight repacking on its own (rt_render_frame_static; rt_set_params does it with the rest) ----
__global__ void repack_kernel(const float* __restrict__ bw, const float* __restrict__ iw, int lf,
                              float* __restrict__ out) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < WPACK_FLOATS) out[e] = packed_value(bw, iw, lf, e);
}

cudaError_t launch_repack(const float* brdf_w, const float* irt_w, int lf, float* wpack, cudaStream_t s) {
  repack_kernel<<<(WPACK_FLOATS + 255) / 256, 256, 0, s>>>(brdf_w, irt_w, lf, wpack);
  return cudaGetLastError();
}

// ---- stage (a) -------------------------------------------------------------
// Thread per (point, level), levels fastest: a point's features are written by
// consecutive lanes (whole 128-byte rows for 16 levels), and a small batch
// still fills the chip.
__global__ void encode_kernel(GridDesc g, const float4* __restrict__ pos, long long PL, float* __restrict__ feat,
                              int feat8, uint32_t* __restrict__ idx, float* __restrict__ wout) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= PL) return;
  const long long p = e / g.levels;
  const int l = (int)(e - p * g.levels);
  const f3 x = xyz(pos[p]);
  const float2 f = encode_level(g, l, x);
  if (feat8) {
    reinterpret_cast<float2*>(feat)[e] = f;
  } else {
    feat[2 * e] = f.x;
    feat[2 * e + 1] = f.y;
  }
  if (idx != nullptr || wout != nullptr) {
    const int res = g.res[l];
    uint32_t ix, iy, iz;
    float wx, wy, wz;
    grid_cell(x.x, res, ix, wx);
    grid_cell(x.y, res, iy, wy);
    grid_cell(x.z, res, iz, wz);
    for (int c = 0; c < 8; ++c) {
      const size_t o = (size_t)e * 8 + c;
      if (idx) idx[o] = corner_row(ix + (c & 1), iy + ((c >> 1) & 1), iz + ((c >> 2) & 1), res, g.dense[l], g.mask);
      if (wout) wout[o] = ((c & 1) ? wx : 1.0f - wx) * ((c & 2) ? wy : 1.0f - wy) * ((c & 4) ? wz : 1.0f - wz);
    }
  }
}

cudaError_t launch_encode(const ModelDesc& m, const float4* pos, int P, float* feat, uint32_t* idx, float* w,
                          cudaStream_t s) {
  const long long PL = (long long)P * m.grid.levels;
  const int feat8 = reinterpret_cast<uintptr_t>(feat) % 8 == 0;
  // P < 2^31 and at most 16 levels: the block count fits the grid's x axis
  encode_kernel<<<(unsigned)((PL + 127) / 128), 128, 0, s>>>(m.grid, pos, PL, feat, feat8, idx, w);
  return cudaGetLastError();
}

// ---- direction sampler -----------------------------------------------------
__global__ void sample_kernel(ModelDesc m, const float4* __restrict__ normal, long long PK, int K, int level,
                              long long offset, float4* __restrict__ dirs) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= PK) return;
  const long long p = e / K;
  const int k = (int)(e % K);
  uint64_t ctr;
  if (level == 0) {
    const uint64_t q = (uint64_t)(offset + p) * (uint64_t)m.N + (uint64_t)k;
    ctr = dir_counter(q, m.M, 0);
  } else {
    ctr = dir_counter((uint64_t)(offset + p), m.M, 1 + k);
  }
  const f3 w = cosine_direction(xyz(normal[p]), m.seed, ctr);
  dirs[e] = make_float4(w.x, w.y, w.z, 0.0f);
}

cudaError_t launch_sample(const ModelDesc& m, const float4* normal, int P, int level, long long offset,
                          float4* dirs, cudaStream_t s) {
  const int K = level == 0 ? m.N : m.M;
  const long long PK = (long long)P * K;
  sample_kernel<<<(unsigned)((PK + 127) / 128), 128, 0, s>>>(m, normal, PK, K, level, offset, dirs);
  return cudaGetLastError();
}

// ---- stage (e) at one level ------------------------------------------------
__global__ void shade_kernel(ModelDesc m, rt_gbuffer pts, int P, int level, long long offset,
                             const float* __restrict__ vis, const float4* __restrict__ lin, float4* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= P) return;
  const f3 n = xyz(reinterpret_cast<const float4*>(pts.normal)[p]);
  const f3 wo = xyz(reinterpret_cast<const float4*>(pts.view)[p]);
  const float4 ar = reinterpret_cast<const float4*>(pts.albedo_rough)[p];
  const f3 alb = xyz(ar);
  const int K = level == 0 ? m.N : m.M;
  f3 acc = mk(0.f, 0.f, 0.f);
  for (int k = 0; k < K; ++k) {
    uint64_t ctr;
    if (level == 0) ctr = dir_counter((uint64_t)(offset + p) * (uint64_t)m.N + (uint64_t)k, m.M, 0);
    else ctr = dir_counter((uint64_t)(offset + p), m.M, 1 + k);
    const f3 w = cosine_direction(n, m.seed, ctr);
    const float v = vis[(size_t)p * K + k];
    f3 li = env_lookup(m.env, m.env_h, m.env_w, w) * v;
    if (lin != nullptr) li = li + xyz(lin[(size_t)p * K + k]) * (1.0f - v);
    acc = acc + li * brdf_eval(alb, ar.w, n, w, wo, m.f0, m.lambert);
  }
  const float sc = kPi / (float)K;
  out[p] = make_float4(acc.x * sc, acc.y * sc, acc.z * sc, 0.0f);
}

cudaError_t launch_shade(const ModelDesc& m, const rt_gbuffer& pts, int P, int level, long long offset,
                         const float* vis, const float4* lin, float4* out, cudaStream_t s) {
  shade_kernel<<<(P + 127) / 128, 128, 0, s>>>(m, pts, P, level, offset, vis, lin, out);
  return cudaGetLastError();
}

cudaError_t prepare_render_fp32();
cudaError_t prepare_render_bf16();
cudaError_t prepare_backward_fp32();
cudaError_t prepare_stages_mlp();

cudaError_t prepare_kernels() {
  cudaError_t e = prepare_render_fp32();
  if (e == cudaSuccess) e = prepare_render_bf16();
  if (e == cudaSuccess) e = prepare_backward_fp32();
  if (e == cudaSuccess) e = prepare_backward_bf16();
  if (e == cudaSuccess) e = prepare_distill();
  if (e == cudaSuccess) e = prepare_stages_mlp();
  return e;
}

}  // namespace rtk
