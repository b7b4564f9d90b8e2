// Per-head distillation of the hash renderer (Sec. 3.3 "Training Procedure";
// supplementary "Training Details"): the stratified whole-sphere directions
// (rt_distill_dirs), the FP32 adjoint of the per-head loss
// (rt_distill_backward) and the Adam update (rt_adam_step).
//
// Loss, for P points x with normals n and K directions each:
//   L1 over B's (n', a', r') against the teacher's, averaged over points and
//   the 7 components; BCE of sigmoid(z0) against the teacher's visibility
//   binarised at 0.5 and L1 of min(softplus(z1), 1) against the teacher's
//   normalised depth, each averaged over the point's front-facing directions
//   (w . n > 0) and then over points.
//
// Work, in two phases of one persistent launch.  I phase: a unit is one
// point and up to 256 of its directions (blocks of 32 in turn); the warp encodes f = H(x), counts
// the point's front-facing directions, lists the unit's (the others carry no
// loss) and walks the list 32 at a time (lane = direction): I forward, the
// head gradients, I's adjoint with the layer-1 f part shared by the unit's
// rows; then it scatters the unit's share of dLoss/df into the table (the
// encode adjoint is linear in it).  Splitting a point's directions over units
// spreads a small batch (2048 points) over every SM.  B phase: a warp takes 32
// points as one 32-row tile (lane = point), runs B, back-propagates the L1 of
// the BRDF heads and scatters the B part of dLoss/df.  Where weight gradients
// are summed: adjoint.cuh.
#include "adjoint.cuh"

namespace rtk {

namespace {

constexpr int kUnitDirs = 256;              // directions of one point per I-phase work unit
// per-warp buffers (floats)
constexpr int DB_F = 0;                                    // f of the warp's 32 points [32 cols]
constexpr int DB_H1 = DB_F + kActStride32;                 // layer-1 activations, then dZ1 (in place) [64 cols]
// PE of the current directions [32 cols] for layer 1, then layer-2 activations and dZ2 (in place)
// [64 cols]; the PE is written again for the PE part of dW1 once dZ2 is consumed
constexpr int DB_H2 = DB_H1 + kActStride;
constexpr int DB_DZ = DB_H2 + kActStride;                 // output gradients [7][32]; column sums [64]
constexpr int DB_FP = DB_DZ + 7 * 32;                      // f of the current point [32]
constexpr int DB_AP = DB_FP + 32;                          // b1 + W1f f of the current point [64]
constexpr int DB_LIST = DB_AP + 64;                        // the unit's front-facing directions, uint16 [256]
constexpr int DB_FLOATS = DB_LIST + kUnitDirs / 2;
constexpr size_t kDSmem = (size_t)(WADJ_FLOATS + kAdjWarps * DB_FLOATS + 4) * sizeof(float);
static_assert(kDSmem <= 232448, "one CTA per SM");
static_assert(DB_H1 % 4 == 0 && DB_H2 % 4 == 0 && DB_H2 == DB_H1 + kActStride && DB_DZ % 4 == 0 &&
                  DB_FLOATS % 4 == 0,
              "float4 alignment");

// Direction j of a point's unit `unit` of nch: the units take blocks of 32 directions in turn.  Stratified directions
// run over the sphere in bands, so a unit of consecutive ones would be all front-facing or all back-facing, and with
// nch dividing the number of warps a warp would meet the same band at every point (2,048 x 1,024: 1.47 ms so, 0.98 ms
// in turn).
__device__ __forceinline__ int unit_dir(int unit, int nch, int j) { return ((unit + nch * (j >> 5)) << 5) + (j & 31); }

// w . n > 0 with every operation pinned: the teacher's and the student's kernels have to agree on it.
__device__ __forceinline__ bool front_facing(float4 w, f3 n) {
  return __fmaf_rn(w.z, n.z, __fmaf_rn(w.y, n.y, __fmul_rn(w.x, n.x))) > 0.0f;
}
__device__ __forceinline__ float sgnf(float d) { return d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f); }

__global__ void distill_dirs_kernel(long long PK, int K, int S, long long ray_offset, uint64_t seed,
                                    float4* __restrict__ dirs) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= PK) return;
  const long long p = e / K;
  const int k = (int)(e - p * K);
  const uint64_t ctr = (uint64_t)(ray_offset + p) * (uint64_t)K + (uint64_t)k;
  const float xi1 = uniform24(splitmix64(seed, 2 * ctr + 1));
  const float xi2 = uniform24(splitmix64(seed, 2 * ctr + 2));
  const float u1 = ((float)(k / S) + xi1) / (float)S;
  const float u2 = ((float)(k % S) + xi2) / (float)S;
  const float z = 1.0f - 2.0f * u1;
  const float rho = 2.0f * sqrtf(fmaxf(u1 * (1.0f - u1), 0.0f));
  float sp, cp;
  sincospif(2.0f * u2, &sp, &cp);
  dirs[e] = make_float4(rho * cp, rho * sp, z, 0.0f);
}

// ---- the teacher's visibility and depth at the front-facing directions ------
// I as the student's kernel evaluates it: FP32 FMA chains in a fixed order, for
// the loss takes signs (hit or not, deeper or not) that a last bit can turn.
// The other directions, half of them on average, have no part in the loss and
// get vis 0 and the near depth: 2,048 x 1,024 take 0.32 ms, rt_trace's
// tensor-core rows over all of them 0.19 ms.  Units and lists as in the I phase;
// one in-place activation buffer per warp, so twelve warps.
constexpr int kTgWarps = 12;
constexpr int kTgThreads = 32 * kTgWarps;
constexpr int TG_ACT = 0, TG_FP = kActStride, TG_AP = TG_FP + 32, TG_LIST = TG_AP + 64;
constexpr int TG_FLOATS = TG_LIST + kUnitDirs / 2;
constexpr size_t kTgSmem = (size_t)(OFF_BW1 + kTgWarps * TG_FLOATS) * sizeof(float);
static_assert(OFF_BW1 % 4 == 0 && TG_FLOATS % 4 == 0 && kTgSmem <= 232448, "float4 alignment, one CTA per SM");

__global__ void __launch_bounds__(kTgThreads, 1)
distill_targets_kernel(ModelDesc m, const float* __restrict__ feat, const float4* __restrict__ dirs,
                       const float4* __restrict__ nrm4, int P, int K, float* __restrict__ vis,
                       float* __restrict__ depth) {
  extern __shared__ float4 smem4[];
  float* sw = reinterpret_cast<float*>(smem4);
  for (int i = threadIdx.x; i < OFF_BW1 / 4; i += kTgThreads) smem4[i] = __ldg(reinterpret_cast<const float4*>(m.wpack) + i);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = lane >> 3, cg = lane & 7;
  float* act = sw + OFF_BW1 + warp * TG_FLOATS + TG_ACT;
  float* fP = act + TG_FP;
  float* aP = act + TG_AP;
  uint16_t* list = reinterpret_cast<uint16_t*>(act + TG_LIST);
  const int nch = (K + kUnitDirs - 1) / kUnitDirs;
  const long long units = (long long)P * nch;
  for (long long u = (long long)blockIdx.x * kTgWarps + warp; u < units; u += (long long)gridDim.x * kTgWarps) {
    const int p = (int)(u / nch);
    const int unit = (int)(u - (long long)p * nch);
    const f3 n = xyz(nrm4[p]);
    fP[lane] = lane < m.lf ? feat[(size_t)p * m.lf + lane] : 0.0f;
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = lane + 32 * h;
      float acc = sw[OFF_IB1 + c];
      for (int k = 0; k < m.lfp; ++k) acc = fmaf(fP[k], sw[OFF_IW1F + k * 64 + c], acc);
      aP[c] = acc;
    }
    int nlist = 0;
#pragma unroll 4
    for (int j0 = 0; unit_dir(unit, nch, j0) < K; j0 += 32) {
      const int k = unit_dir(unit, nch, j0 + lane);
      const bool ff = k < K && front_facing(dirs[(size_t)p * K + k], n);
      if (k < K && !ff) {
        vis[(size_t)p * K + k] = 0.0f;
        depth[(size_t)p * K + k] = m.near_t;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, ff);
      if (ff) list[nlist + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(j0 + lane);
      nlist += __popc(bal);
    }
    __syncwarp();
    for (int r0 = 0; r0 < nlist; r0 += 32) {
      const bool ff = r0 + lane < nlist;
      const size_t e = (size_t)p * K + unit_dir(unit, nch, (int)list[ff ? r0 + lane : r0]);
      Tile acc;
      store_pe(act, xyz(dirs[e]), lane);
      __syncwarp();
      zero(acc);
      warp_gemm<kPEPad - 4>(act, sw + OFF_IW1P, acc, rg, cg);
      __syncwarp();
      store_relu_colbias(act, acc, aP, rg, cg);
      __syncwarp();
      zero(acc);
      warp_gemm<kHidden>(act, sw + OFF_IW2, acc, rg, cg);
      __syncwarp();
      store_relu_colbias(act, acc, sw + OFF_IB2, rg, cg);
      __syncwarp();
      const float2 z = irt_head(act, sw, lane);
      if (ff) {
        vis[e] = sigmoidf_(z.x);
        depth[e] = depth_from_logit(z.y, m.near_t, m.far_t);
      }
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(kAdjThreads, 1)
distill_fp32_kernel(ModelDesc m, const float4* __restrict__ pos4, const float4* __restrict__ nrm4, int P, int K,
                    const float4* __restrict__ dirs, const float* __restrict__ brdf_t, const float* __restrict__ vis_t,
                    const float* __restrict__ depth_t, float* __restrict__ loss, float* __restrict__ g_table,
                    float* __restrict__ g_brdf, float* __restrict__ g_irt) {
  extern __shared__ float4 smem4[];
  float* sw = reinterpret_cast<float*>(smem4);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sw + WADJ_FLOATS + kAdjWarps * DB_FLOATS);
  load_adjoint_weights(sw, m.wpack);
  const uint32_t tacc = adj_tmem_alloc(tslot, threadIdx.x);   // (its barrier also publishes the weights)
  tmem_zero(tacc, 12);
  IrtGrads gI;
  zero(gI);
  const float* bw = m.wpack;   // B's weights stay in global memory (one evaluation per point)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rg = lane >> 3, cg = lane & 7;
  float* wb = sw + WADJ_FLOATS + warp * DB_FLOATS;
  float* F = wb + DB_F;
  float* PEb = wb + DB_H2;   // shares H2's buffer (see DB_H2)
  float* H1 = wb + DB_H1;
  float* H2 = wb + DB_H2;
  float* DZ = wb + DB_DZ;
  float* fP = wb + DB_FP;
  float* aP = wb + DB_AP;
  uint16_t* list = reinterpret_cast<uint16_t*>(wb + DB_LIST);
  const int lf = m.lf, lfp = m.lfp, levels = m.grid.levels;
  const BlobB gB{g_brdf, lf};
  const float invR = 1.0f / (float)P;
  const float inv_range = 1.0f / (m.far_t - m.near_t);
  float l_brdf = 0.0f, l_bce = 0.0f, l_depth = 0.0f;

  // ---- I phase: units of (point, up to kUnitDirs of its directions), lane = direction
  const int nch = (K + kUnitDirs - 1) / kUnitDirs;
  const long long units = (long long)P * nch;
  for (long long u = (long long)blockIdx.x * kAdjWarps + warp; u < units; u += (long long)gridDim.x * kAdjWarps) {
    {
      const int p = (int)(u / nch);
      const int unit = (int)(u - (long long)p * nch);
      const f3 x = xyz(pos4[p]);
      const f3 n = xyz(nrm4[p]);
      {
        const int l = lane >> 1;
        float2 part = make_float2(0.f, 0.f);
        if (l < levels) {
          const float2 f = encode_level_exact(m.grid, l, x);
          part = (lane & 1) ? make_float2(0.f, 0.f) : f;
        }
        if ((lane & 1) == 0) {
          fP[lane] = part.x;
          fP[lane + 1] = part.y;
        }
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = lane + 32 * h;
        float acc = sw[OFF_IB1 + c];
        for (int k = 0; k < lfp; ++k) acc = fmaf(fP[k], sw[OFF_IW1F + k * 64 + c], acc);
        aP[c] = acc;
      }
      // the point's front-facing count, and the unit's front-facing directions in order: the others have no
      // part in the loss, so only these are evaluated
      int cnt = 0, nlist = 0;
#pragma unroll 4   // the loads of four steps in flight
      for (int k0 = 0; k0 < K; k0 += 32) {
        const int k = k0 + lane;
        const bool ff = k < K && front_facing(dirs[(size_t)p * K + k], n);
        const unsigned bal = __ballot_sync(0xffffffffu, ff);
        cnt += __popc(bal);
        if ((k0 >> 5) % nch == unit) {
          if (ff) list[nlist + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)(((k0 >> 5) / nch << 5) + lane);
          nlist += __popc(bal);
        }
      }
      const float wI = cnt > 0 ? invR / (float)cnt : 0.0f;
      float cs[2] = {0.f, 0.f};   // the unit's sum of dZ1, the lane's two columns
      __syncwarp();
      for (int r0 = 0; r0 < nlist; r0 += 32) {
        const bool ff = r0 + lane < nlist;
        const int k = unit_dir(unit, nch, (int)list[ff ? r0 + lane : r0]);
        const f3 w = xyz(dirs[(size_t)p * K + k]);
        Tile acc;
        store_pe(PEb, w, lane);
        __syncwarp();
        zero(acc);
        warp_gemm<kPEPad - 4>(PEb, sw + OFF_IW1P, acc, rg, cg);
        store_relu_colbias(H1, acc, aP, rg, cg);
        __syncwarp();
        zero(acc);
        warp_gemm<kHidden>(H1, sw + OFF_IW2, acc, rg, cg);
        store_relu_colbias(H2, acc, sw + OFF_IB2, rg, cg);
        __syncwarp();
        const float2 z = irt_head(H2, sw, lane);
        float dz0 = 0.0f, dz1 = 0.0f;
        if (ff) {
          const size_t e = (size_t)p * K + k;
          const float vt = vis_t[e] > 0.5f ? 1.0f : 0.0f;
          const float dt = (depth_t[e] - m.near_t) * inv_range;
          l_bce += wI * (fmaxf(z.x, 0.0f) - z.x * vt + log1pf(expf(-fabsf(z.x))));
          dz0 = wI * (sigmoidf_(z.x) - vt);
          const float sp = softplusf_(z.y);
          const float d = fminf(sp, 1.0f) - dt;
          l_depth += wI * fabsf(d);
          dz1 = sp < 1.0f ? wI * sgnf(d) * sigmoidf_(z.y) : 0.0f;
        }
        DZ[lane] = dz0;
        DZ[32 + lane] = dz1;
        gI.b3[0] += dz0;
        gI.b3[1] += dz1;
        __syncwarp();
        bwd_out<2>(H2, DZ, sw + OFF_IW3, gI.w3, gI.b2, lane);
        __syncwarp();
        acc_w2(H1, H2, tacc, rg, cg);
        bwd_hidden_tile(H2, sw + OFF_IW2T, H1, acc, rg, cg);
        store_pe(PEb, w, lane);   // again, over the consumed dZ2
        __syncwarp();
        acc_w1p(PEb, H1, tacc, rg, cg);
        col_sums(H1, cs, lane);   // the f part of layer 1 is shared by the unit's rows: once per unit, below
        __syncwarp();
      }
      if (nlist > 0) {
        DZ[own_col(lane, 0)] = cs[0];
        DZ[own_col(lane, 1)] = cs[1];
        gI.b1[0] += cs[0];
        gI.b1[1] += cs[1];
        __syncwarp();
        const float dfk = bwd_shared_feature(fP, DZ, sw + OFF_IW1F, lf, g_irt, lane);
        // the unit's share of dLoss/df (the encode adjoint is linear in it)
        const int l = lane >> 1;
        const float df1 = __shfl_down_sync(0xffffffffu, dfk, 1);
        if ((lane & 1) == 0 && l < levels) encode_level_bwd(m.grid, l, x, dfk, df1, g_table, nullptr);
      }
      __syncwarp();
    }
  }

  // ---- B phase: groups of 32 points as one 32-row tile (lane = point), from the last warp on: the first ones may
  // have had one unit more
  for (long long g0 = ((long long)(gridDim.x - blockIdx.x) * kAdjWarps - 1 - warp) * 32; g0 < P;
       g0 += (long long)gridDim.x * kAdjWarps * 32) {
    const int p = (int)min(g0 + lane, (long long)P);
    const bool vp = p < P;
    {
      const f3 x = vp ? xyz(pos4[p]) : mk(0.f, 0.f, 0.f);
#pragma unroll 1
      for (int l = 0; l < kMaxLevels; ++l) {
        const float2 f = (vp && l < levels) ? encode_level_exact(m.grid, l, x) : make_float2(0.f, 0.f);
        F[aidx(2 * l, lane)] = f.x;
        F[aidx(2 * l + 1, lane)] = f.y;
      }
    }
    __syncwarp();
    Tile acc;
    zero(acc);
    warp_gemm_k(F, bw + OFF_BW1, acc, lfp, rg, cg);
    store_relu_colbias(H1, acc, bw + OFF_BB1, rg, cg);
    __syncwarp();
    zero(acc);
    warp_gemm<kHidden>(H1, bw + OFF_BW2, acc, rg, cg);
    store_relu_colbias(H2, acc, bw + OFF_BB2, rg, cg);
    __syncwarp();
    float y[7];
#pragma unroll
    for (int o = 0; o < 7; ++o) y[o] = __ldg(bw + OFF_BB3 + o);
    for (int k = 0; k < kHidden; ++k) {
      const float hk = H2[aidx(k, lane)];
#pragma unroll
      for (int o = 0; o < 7; ++o) y[o] = fmaf(hk, __ldg(bw + OFF_BW3 + 8 * k + o), y[o]);
    }
    const float nlen = sqrtf(fmaxf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2], 1e-24f));
    const f3 n2 = mk(y[0] / nlen, y[1] / nlen, y[2] / nlen);
    const f3 a2 = mk(sigmoidf_(y[3]), sigmoidf_(y[4]), sigmoidf_(y[5]));
    const float s6 = sigmoidf_(y[6]);
    const float r2 = 0.09f + 0.91f * s6;
    float dy[7];
    {
      const float wB = vp ? invR / 7.0f : 0.0f;
      float t[7];
#pragma unroll
      for (int o = 0; o < 7; ++o) t[o] = vp ? brdf_t[(size_t)p * 8 + o] : 0.0f;
      const float out[7] = {n2.x, n2.y, n2.z, a2.x, a2.y, a2.z, r2};
      float g[7];
#pragma unroll
      for (int o = 0; o < 7; ++o) {
        l_brdf += wB * fabsf(out[o] - t[o]);
        g[o] = wB * sgnf(out[o] - t[o]);
      }
      const f3 dn = mk(g[0], g[1], g[2]);
      const float dnn = dot(n2, dn);
      dy[0] = (dn.x - n2.x * dnn) / nlen;
      dy[1] = (dn.y - n2.y * dnn) / nlen;
      dy[2] = (dn.z - n2.z * dnn) / nlen;
      dy[3] = g[3] * a2.x * (1.0f - a2.x);
      dy[4] = g[4] * a2.y * (1.0f - a2.y);
      dy[5] = g[5] * a2.z * (1.0f - a2.z);
      dy[6] = g[6] * 0.91f * s6 * (1.0f - s6);
    }
#pragma unroll
    for (int o = 0; o < 7; ++o) DZ[o * 32 + lane] = dy[o];
    __syncwarp();
    bwd_w3<7>(H2, DZ, gB.w3(), gB.b3(), lane, 64);
    __syncwarp();
    bwd_head<7, 8>(H2, DZ, bw + OFF_BW3, H2, lane);   // dZ2 over H2, in place
    __syncwarp();
    bwd_weights_global(H1, 64, H2, gB.w2(), 64, gB.b2(), lane);
    __syncwarp();
    bwd_hidden(H2, bw + OFF_BW2, H1, H1, lane);   // dZ1 over H1, in place
    __syncwarp();
    bwd_weights_global(F, lf, H1, gB.w1(), lf, gB.b1(), lane);
    float dF[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) dF[k] = 0.0f;
    bwd_input(H1, bw + OFF_BW1, lf, dF, lane);
    {
      // segmented scatter over the warp's points (Morton order, runs of equal rows summed first)
      uint32_t dbits[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) dbits[k] = __float_as_uint(dF[k]);
      const f3 x = vp ? xyz(pos4[p]) : mk(0.f, 0.f, 0.f);
      (void)encode_bwd_sorted<false>(m.grid, x, dbits, vp, g_table, nullptr);
    }
    __syncwarp();
  }

  // ---- loss terms (one atomic per warp) and the weight gradients
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    l_brdf += __shfl_xor_sync(0xffffffffu, l_brdf, o);
    l_bce += __shfl_xor_sync(0xffffffffu, l_bce, o);
    l_depth += __shfl_xor_sync(0xffffffffu, l_depth, o);
  }
  if (lane == 0 && loss != nullptr) {
    atomicAdd(loss + 0, l_brdf);
    atomicAdd(loss + 1, l_bce);
    atomicAdd(loss + 2, l_depth);
  }
  flush_irt_grads(sw + WADJ_FLOATS + DB_H1, DB_FLOATS, tacc, gI, lf, g_irt);
  adj_tmem_free(tslot, threadIdx.x);
}

struct AdamConst {
  float lr, b1, b2, eps, wd, bc1, bc2;
};
__device__ __forceinline__ void adam_one(float& p, float g, float& m1, float& m2, const AdamConst& k) {
  const float gg = g + k.wd * p;
  m1 = k.b1 * m1 + (1.0f - k.b1) * gg;
  m2 = k.b2 * m2 + (1.0f - k.b2) * gg * gg;
  p -= k.lr * (m1 / k.bc1) / (sqrtf(m2 / k.bc2) + k.eps);
}

// Elementwise, 28 bytes of traffic per parameter: bound by HBM.  n4 groups of four values as 16-byte accesses (buffers
// 16-byte aligned), then the rest one by one, which is all of them where a buffer is a slice at an odd offset.
// 30 M parameters: 133 us, 199 us by 4-byte accesses with four elements' loads in flight (269 us one at a time).
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                            float* __restrict__ m2, long long n4, long long n, AdamConst k) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, stride = (long long)gridDim.x * blockDim.x;
  for (long long e = i; e < n4; e += stride) {
    float4 pv = reinterpret_cast<float4*>(p)[e], a = reinterpret_cast<float4*>(m1)[e], b = reinterpret_cast<float4*>(m2)[e];
    const float4 gv = reinterpret_cast<const float4*>(g)[e];
    adam_one(pv.x, gv.x, a.x, b.x, k);
    adam_one(pv.y, gv.y, a.y, b.y, k);
    adam_one(pv.z, gv.z, a.z, b.z, k);
    adam_one(pv.w, gv.w, a.w, b.w, k);
    reinterpret_cast<float4*>(m1)[e] = a;
    reinterpret_cast<float4*>(m2)[e] = b;
    reinterpret_cast<float4*>(p)[e] = pv;
  }
#pragma unroll 4   // independent elements: the loads of four in flight
  for (long long e = 4 * n4 + i; e < n; e += stride) {
    float pv = p[e], a = m1[e], b = m2[e];
    adam_one(pv, g[e], a, b, k);
    m1[e] = a;
    m2[e] = b;
    p[e] = pv;
  }
}

}  // namespace

cudaError_t prepare_distill() {
  const cudaError_t e =
      cudaFuncSetAttribute(distill_targets_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTgSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(distill_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDSmem);
}

cudaError_t launch_distill_dirs(int P, int K, long long ray_offset, uint64_t seed, float4* dirs, cudaStream_t s) {
  int S = 1;
  while ((S + 1) * (S + 1) <= K) ++S;
  const long long PK = (long long)P * K;
  distill_dirs_kernel<<<(unsigned)((PK + 255) / 256), 256, 0, s>>>(PK, K, S, ray_offset, seed, dirs);
  return cudaGetLastError();
}

cudaError_t launch_distill_targets(const ModelDesc& m, const float* feat, const float4* dirs, const float4* nrm, int P,
                                   int K, float* vis, float* depth, int num_sms, cudaStream_t s) {
  const long long units = (long long)P * ((K + kUnitDirs - 1) / kUnitDirs);
  const long long need = (units + kTgWarps - 1) / kTgWarps;
  const int grid = (int)(need < num_sms ? need : num_sms);
  distill_targets_kernel<<<grid, kTgThreads, kTgSmem, s>>>(m, feat, dirs, nrm, P, K, vis, depth);
  return cudaGetLastError();
}

cudaError_t launch_distill_fp32(const ModelDesc& m, const float4* pos, const float4* nrm, int P, int K,
                                const float4* dirs, const float* brdf_t, const float* vis_t, const float* depth_t,
                                float* loss, float* g_table, float* g_brdf, float* g_irt, int num_sms, cudaStream_t s) {
  const long long units = (long long)P * ((K + kUnitDirs - 1) / kUnitDirs);
  const long long groups = (P + 31) / 32;
  const long long need = ((units > groups ? units : groups) + kAdjWarps - 1) / kAdjWarps;
  const int grid = (int)(need < num_sms ? need : num_sms);
  distill_fp32_kernel<<<grid, kAdjThreads, kDSmem, s>>>(m, pos, nrm, P, K, dirs, brdf_t, vis_t, depth_t, loss, g_table,
                                                g_brdf, g_irt);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* p, const float* g, float* m1, float* m2, long long n, float lr, float b1, float b2,
                        float eps, float wd, float bc1, float bc2, int num_sms, cudaStream_t s) {
  const uintptr_t bits = reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(g) | reinterpret_cast<uintptr_t>(m1) |
                         reinterpret_cast<uintptr_t>(m2);
  const long long n4 = bits % 16 == 0 ? n / 4 : 0;
  const long long blocks = ((n4 > 0 ? (n + 3) / 4 : n) + 255) / 256;
  const int grid = (int)(blocks < 8LL * num_sms ? blocks : 8LL * num_sms);
  adam_kernel<<<grid > 0 ? grid : 1, 256, 0, s>>>(p, g, m1, m2, n4, n, AdamConst{lr, b1, b2, eps, wd, bc1, bc2});
  return cudaGetLastError();
}

}  // namespace rtk
