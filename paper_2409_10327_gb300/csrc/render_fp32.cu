// Fused FP32 hot path: stages (a)-(e) of the hash renderer in one persistent
// kernel (rt_render_frame with precision RT_FP32).
//
// Work unit: a warpgroup owns a contiguous range of primary points and walks
// its (point, direction) samples in tiles of 128 consecutive ones; thread t of
// the warpgroup owns row t of the tile, which is TMEM lane t.
//
// Two kinds of MLP evaluation.  I(f, w_i) and B(f') decide x' and the shading
// frame there: a changed last bit of t moves x' across the finest cells and a
// sharp lobe, and reaches single pixels enlarged a thousandfold.  They run as
// FP32 FMA chains in a fixed order (warp_gemm.cuh: each warp its 32 rows).
// The M evaluations I(f', w'_j), four fifths of the arithmetic, only yield
// visibilities, which pass their rounding on as it is: they are tcgen05.mma
// chains on three-part bf16 operands (tc_split.cuh), which carry FP32's 24
// significant bits.  Everything else is FP32 on the CUDA cores.  Two
// warpgroups share a CTA; while one waits for its tensor-core chain the other
// computes, and within a warpgroup the BRDF and environment lookup of a
// direction overlap its layer 1, and the next direction and its encoding
// overlap its layer 2.
// 800 x 800 x 128 directions: 133 ms, 247 ms with every evaluation on the FMA
// pipes; 97 x 61 x 40 (consecutive rows instead of 32 directions of one pixel
// per warp, which wasted three rows in eight there): 422 us, 1,164 us.
//
// TMEM columns of a warpgroup (256 from column 256 * wg):
//   D [0, 64)     FP32 accumulator of both layers
//   X [64, 160)   layer-1 input [f' (32) | PE (27) | 1 1 1 0 0], three parts of 32 columns
//   H [160, 256)  layer-2 input relu(layer 1), three parts
//
// A pixel's sum does not depend on how tiles fall on it: lane k of a warp adds
// the contributions i = k (mod 32) in order of i, carried over tiles in shared
// memory, then a butterfly adds the lanes.  So a frame rendered in shards has
// the same bits as in one call.
#include "mis.cuh"
#include "tc_split.cuh"
#include "warp_gemm.cuh"

namespace rtk {

namespace {

constexpr int kWG = 2;
constexpr int kThreads = 128 * kWG;
constexpr int kTmemCols = 256 * kWG;
constexpr int TM_D = 0, TM_X = 64, TM_H = 160;
constexpr int kSlots = 10;       // pixels of a tile whose feature part of layer 1 is shared (N >= 16)
// shared memory from a 1024-aligned base: I's split weights (parts, layer-2 bias, ones), the packed FP32 image, I's
// visibility row, an activation buffer per warp, then per warpgroup
constexpr int SM_W1 = 0, SM_W2 = 3 * kPart, SM_B2 = 6 * kPart, SM_ONES = SM_B2 + 2048;
constexpr int SM_W = SM_ONES + 4096;                  // float [WPACK_FLOATS - OFF_IW1P]: the packed image from I's PE rows on
constexpr int SM_HV = SM_W + (WPACK_FLOATS - OFF_IW1P) * 4;        // float [64]
constexpr int SM_ACT = SM_HV + 64 * 4;                // float [8 warps][kActStride]
constexpr int SM_WG = SM_ACT + 4 * kWG * kActStride * 4;
constexpr int WG_AP = 0;                              // float [kSlots][64]: b1 + W1f f of the tile's pixels
constexpr int WG_RED = WG_AP + kSlots * 64 * 4;    // float4 [128]: the tile's contributions
constexpr int WG_CARRY = WG_RED + 128 * 16;           // float4 [2][32]: lane sums of a pixel that continues, by tile parity
constexpr int WG_BAR = WG_CARRY + 2 * 32 * 16;        // mbarrier
constexpr int WG_BYTES = WG_BAR + 16;
constexpr int kTmemSlot = SM_WG + kWG * WG_BYTES;
constexpr size_t kSmemBytes = kTmemSlot + 16 + 1024;
static_assert(SM_W % 16 == 0 && SM_HV % 16 == 0 && SM_ACT % 16 == 0 && SM_WG % 16 == 0 && WG_RED % 16 == 0 &&
                  WG_BYTES % 16 == 0,
              "aligned blocks");
// The gathers of the x' encode live on L1: a line of it per lane and corner.  One step of the shared-memory
// configurations below the largest leaves 60 KB of the SM for L1 instead of 28 KB: 150 -> 133 ms for the frame above.
static_assert(kSmemBytes + 1024 <= 196 * 1024, "fits the 196 KB configuration");

// Four corners of level l's cell at x (corners 4 half .. 4 half + 3) weighted and summed; a level's primary feature
// is the sum of its two halves.
__device__ __forceinline__ float2 encode_half(const GridDesc& g, int l, int half, f3 x) {
  const int res = g.res[l];
  uint32_t ix, iy, iz;
  float wx, wy, wz;
  grid_cell_exact(x.x, res, ix, wx);
  grid_cell_exact(x.y, res, iy, wy);
  grid_cell_exact(x.z, res, iz, wz);
  const size_t base = (size_t)l << g.log2T;
  float2 part = make_float2(0.f, 0.f);
#pragma unroll
  for (int cc = 0; cc < 4; ++cc) {
    const int c = half * 4 + cc;
    const uint32_t row = corner_row(ix + (c & 1), iy + ((c >> 1) & 1), iz + ((c >> 2) & 1), res, g.dense[l], g.mask);
    const float w = ((c & 1) ? wx : 1.0f - wx) * ((c & 2) ? wy : 1.0f - wy) * ((c & 4) ? wz : 1.0f - wz);
    const float2 v = table_entry(g, base + row);
    part.x = fmaf(w, v.x, part.x);
    part.y = fmaf(w, v.y, part.y);
  }
  return part;
}

// (a) f = H(x) of one pixel (lanes 2l and 2l + 1 take half of level l each), then I's layer-1 bias b1 + W1f f, shared
// by the pixel's directions, into aP [64]; fP: 32 floats of the warp's scratch.
__device__ __forceinline__ void primary_bias(const GridDesc& g, f3 x, const float* __restrict__ wpack, int lfp,
                                             float* fP, float* aP, int lane) {
  float2 part = make_float2(0.f, 0.f);
  if ((lane >> 1) < g.levels) part = encode_half(g, lane >> 1, lane & 1, x);
  part.x += __shfl_xor_sync(0xffffffffu, part.x, 1);
  part.y += __shfl_xor_sync(0xffffffffu, part.y, 1);
  if ((lane & 1) == 0) {
    fP[lane] = part.x;
    fP[lane + 1] = part.y;
  }
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int c = lane + 32 * h;
    float acc = __ldg(wpack + OFF_IB1 + c);
#pragma unroll 8
    for (int k = 0; k < lfp; ++k) acc = fmaf(fP[k], __ldg(wpack + OFF_IW1F + k * 64 + c), acc);
    aP[c] = acc;
  }
  __syncwarp();
}

// act(col, row) = relu(t + aP[slot of the row][col]); slot: this lane's row's
__device__ __forceinline__ void store_relu_slotbias(float* __restrict__ act, const Tile& t, const float* aP, int slot,
                                                    int rg, int cg) {
  if (__all_sync(0xffffffffu, slot == __shfl_sync(0xffffffffu, slot, 0))) {
    store_relu_colbias(act, t, aP + slot * 64, rg, cg);
    return;
  }
  Tile bias;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float* b0 = aP + __shfl_sync(0xffffffffu, slot, 8 * rg + 2 * q) * 64;
    const float* b1 = aP + __shfl_sync(0xffffffffu, slot, 8 * rg + 2 * q + 1) * 64;
#pragma unroll
    for (int c = 0; c < 8; ++c) bias.v[q][c] = make_float2(b0[ocol(cg, c)], b1[ocol(cg, c)]);
  }
  store_relu_tilebias(act, t, bias, rg, cg);
}

// a 64-wide layer over the warp's rows in place: act = relu(act W + b)
__device__ __forceinline__ void layer_in_place(float* act, const float* W, const float* b, int rg, int cg) {
  Tile t;
  zero(t);
  warp_gemm<kHidden>(act, W, t, rg, cg);
  __syncwarp();
  store_relu_colbias(act, t, b, rg, cg);
  __syncwarp();
}

__global__ void __launch_bounds__(kThreads, 1)
render_fp32_kernel(const __grid_constant__ ModelDesc m, rt_gbuffer gb, int P, long long pixel_offset,
                   float4* __restrict__ out) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x;
  const int wg = __shfl_sync(0xffffffffu, tid >> 7, 0), t = tid & 127, warp = __shfl_sync(0xffffffffu, t >> 5, 0), lane = t & 31;
  const int rg = lane >> 3, cg = lane & 7;
  uint8_t* wgb = sm + SM_WG + wg * WG_BYTES;
  float* aP = reinterpret_cast<float*>(wgb + WG_AP);
  float4* red = reinterpret_cast<float4*>(wgb + WG_RED);
  float4* carry = reinterpret_cast<float4*>(wgb + WG_CARRY);
  const float* sw = reinterpret_cast<const float*>(sm + SM_W) - OFF_IW1P;   // indexed like the packed image
  float* hv = reinterpret_cast<float*>(sm + SM_HV);
  float* act = reinterpret_cast<float*>(sm + SM_ACT) + (tid >> 5) * kActStride;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kTmemSlot);
  const uint32_t bar = smem_u32(wgb + WG_BAR);

  // ---- CTA set-up: split weights into shared memory, TMEM, barriers
  build_split_matrix(sm + SM_W1, m.wpack + OFF_IW1F, 32 + kPE, m.wpack + OFF_IB1, tid, kThreads);
  build_split_matrix(sm + SM_W2, m.wpack + OFF_IW2, 64, nullptr, tid, kThreads);
  build_split_bias(sm + SM_B2, m.wpack + OFF_IB2, tid, kThreads);
  build_split_ones(sm + SM_ONES, tid, kThreads);
  static_assert(OFF_IW1P % 4 == 0, "float4 copy");
  for (int i = tid; i < (WPACK_FLOATS - OFF_IW1P) / 4; i += kThreads)
    reinterpret_cast<float4*>(sm + SM_W)[i] = __ldg(reinterpret_cast<const float4*>(m.wpack + OFF_IW1P) + i);
  if (tid < 64) hv[tid] = __ldg(m.wpack + OFF_IW3 + 2 * tid);
  if (t == 0) {
    mbar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_async_smem();   // the weight tiles are read by the async proxy
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0) + (uint32_t)(256 * wg);
  const uint32_t D_t = tmem + TM_D, X_t = tmem + TM_X, H_t = tmem + TM_H;   // MMA operands (lane 0)
  const uint32_t lane_off = (uint32_t)(32 * warp) << 16;                    // this warp's 32 lanes
  const uint32_t D_w = D_t + lane_off, X_w = X_t + lane_off, H_w = H_t + lane_off;
  const uint32_t S = smem_u32(sm);

  const int N = m.N, M = m.M, lfp = m.lfp;
  const float4* pos4 = reinterpret_cast<const float4*>(gb.pos);
  const float4* nrm4 = reinterpret_cast<const float4*>(gb.normal);
  const float4* view4 = reinterpret_cast<const float4*>(gb.view);
  const float4* ar4 = reinterpret_cast<const float4*>(gb.albedo_rough);

  const long long workers = (long long)gridDim.x * kWG;
  const long long worker = (long long)blockIdx.x * kWG + wg;
  const long long p0 = (long long)P * worker / workers, p1 = (long long)P * (worker + 1) / workers;
  const long long s_end = p1 * N;
  uint32_t phase = 0, pending_phase = 0;
  int abort = 0;

  // An MMA chain in two halves: issue (a barrier with an abort vote, then one
  // thread issues and commits) and a bounded wait.  A wait that gives up only
  // raises `abort`; the vote at the next issue then stops all 128 threads
  // together, so the warpgroup never splits across barriers.
  auto issue = [&](auto chain) -> bool {
    tmem_st_wait();   // this thread's rows of the A operand have landed in TMEM
    tc_fence_before();
    abort = wg_sync_or(wg, abort);
    if (abort) return false;
    if (warp == 0) {
      const uint32_t one = elect_one();
      tc_fence_after();
      chain(one);
      mma_commit(one, bar);
      __syncwarp();
    }
    return true;
  };
  auto wait = [&] {
    if (!mbar_wait(bar, phase)) {
      if (!abort && t == 0) atomicOr(m.status, kStatusTimeout | kWhereRenderFp32);
      abort = 1;
      pending_phase = phase;
    }
    phase ^= 1u;
    tc_fence_after();
  };
  auto irt_layer1 = [&] { return issue([&](uint32_t one) { mma_split3<0, 4>(one, D_t, X_t, S + SM_W1); }); };
  auto irt_layer2 = [&] { return issue([&](uint32_t one) { mma_split3_layer2(one, D_t, H_t, S + SM_W2, S + SM_ONES, S + SM_B2); }); };

  uint32_t parity = 0;
  for (long long sbase = p0 * N; sbase < s_end; sbase += 128, parity ^= 1u) {
    const long long p_first = sbase / N;
    const int off0 = (int)(sbase - p_first * N);
    const int nvalid = (int)min(128LL, s_end - sbase);
    const int npix = (int)((sbase + nvalid - 1) / N - p_first) + 1;
    const bool valid = t < nvalid;
    const int local = off0 + (valid ? t : nvalid - 1);   // idle rows repeat the last sample
    const int ps = local / N;
    const int i = local - ps * N;
    const long long p = p_first + ps;
    const f3 x = xyz(pos4[p]);
    const f3 n = xyz(nrm4[p]);
    const f3 wo = xyz(view4[p]);
    const float4 ar = ar4[p];

    const uint64_t q = (uint64_t)(pixel_offset + p) * (uint64_t)N + (uint64_t)i;
    const f3 wi = m.mis ? mis_direction(m, n, wo, ar.w, i, dir_counter(q, M, 0))
                        : cosine_direction(n, m.seed, dir_counter(q, M, 0));

    // (a) and (c) I(f, w_i).  The feature part of layer 1 once per pixel; per row where a tile may span more pixels
    // than there are slots (N < 16)
    Tile acc;
    if (npix <= kSlots) {
      for (int s = warp; s < npix; s += 4) primary_bias(m.grid, xyz(pos4[p_first + s]), m.wpack, lfp, act, aP + 64 * s, lane);
      wg_sync(wg);
      store_pe(act, wi, lane);
      __syncwarp();
      zero(acc);
      warp_gemm<kPEPad - 4>(act, sw + OFF_IW1P, acc, rg, cg);
      __syncwarp();
      store_relu_slotbias(act, acc, aP, ps, rg, cg);
    } else {
      for (int l = 0; l < kMaxLevels; ++l) {
        float2 f = make_float2(0.f, 0.f);
        if (l < m.grid.levels) {
          const float2 f0 = encode_half(m.grid, l, 0, x), f1 = encode_half(m.grid, l, 1, x);
          f = make_float2(f0.x + f1.x, f0.y + f1.y);
        }
        act[aidx(2 * l, lane)] = f.x;
        act[aidx(2 * l + 1, lane)] = f.y;
      }
      __syncwarp();
      Tile bias;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const float b = sw[OFF_IB1 + ocol(cg, c)];
#pragma unroll
        for (int r = 0; r < 4; ++r) bias.v[r][c] = make_float2(b, b);
      }
      warp_gemm_k(act, m.wpack + OFF_IW1F, bias, lfp, rg, cg);
      __syncwarp();
      store_pe(act, wi, lane);
      __syncwarp();
      zero(acc);
      warp_gemm<kPEPad - 4>(act, sw + OFF_IW1P, acc, rg, cg);
      __syncwarp();
      store_relu_tilebias(act, acc, bias, rg, cg);
    }
    __syncwarp();
    layer_in_place(act, sw + OFF_IW2, sw + OFF_IB2, rg, cg);
    const float2 z = irt_head(act, sw, lane);
    const float v = visibility_from_logit(z.x, m.force_vis, m.hard);
    const float tdep = depth_from_logit(z.y, m.near_t, m.far_t);
    __syncwarp();

    // (d) bounce: x' = x + t w_i, f' = H(x'), for B as it is and for I in parts
    const f3 x2 = x + wi * tdep;
#pragma unroll 1
    for (int it = 0; it < kMaxLevels / 4; ++it) {
      uint32_t q0[4], q1[4], q2[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int l = 4 * it + b;
        float2 f = make_float2(0.f, 0.f);
        if (l < m.grid.levels) f = encode_level_exact(m.grid, l, x2);
        act[aidx(2 * l, lane)] = f.x;
        act[aidx(2 * l + 1, lane)] = f.y;
        split3(f.x, f.y, q0[b], q1[b], q2[b]);
      }
      tmem_st4(X_w + 4 * it, q0[0], q0[1], q0[2], q0[3]);
      tmem_st4(X_w + 32 + 4 * it, q1[0], q1[1], q1[2], q1[3]);
      tmem_st4(X_w + 64 + 4 * it, q2[0], q2[1], q2[2], q2[3]);
    }
    __syncwarp();

    // (b) B(f')
    zero(acc);
    warp_gemm_k(act, sw + OFF_BW1, acc, lfp, rg, cg);
    __syncwarp();
    store_relu_colbias(act, acc, sw + OFF_BB1, rg, cg);
    __syncwarp();
    layer_in_place(act, sw + OFF_BW2, sw + OFF_BB2, rg, cg);
    float y[7];
#pragma unroll
    for (int o = 0; o < 7; ++o) y[o] = sw[OFF_BB3 + o];
#pragma unroll 4
    for (int k = 0; k < kHidden; ++k) {
      const float h = act[aidx(k, lane)];
      const float4 w0 = *reinterpret_cast<const float4*>(sw + OFF_BW3 + 8 * k);
      const float4 w1 = *reinterpret_cast<const float4*>(sw + OFF_BW3 + 8 * k + 4);
      y[0] = fmaf(h, w0.x, y[0]);
      y[1] = fmaf(h, w0.y, y[1]);
      y[2] = fmaf(h, w0.z, y[2]);
      y[3] = fmaf(h, w0.w, y[3]);
      y[4] = fmaf(h, w1.x, y[4]);
      y[5] = fmaf(h, w1.y, y[5]);
      y[6] = fmaf(h, w1.z, y[6]);
    }
    __syncwarp();   // the buffer is free for the next tile
    const float ninv = rsqrtf(fmaxf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2], 1e-24f));
    const f3 n2 = mk(y[0] * ninv, y[1] * ninv, y[2] * ninv);
    const f3 a2 = mk(sigmoidf_(y[3]), sigmoidf_(y[4]), sigmoidf_(y[5]));
    const float r2 = 0.09f + 0.91f * sigmoidf_(y[6]);
    const f3 wo2 = neg(wi);

    // (c) + (e) at x': M directions about n'
    f3 lo2 = mk(0.f, 0.f, 0.f);
    f3 wj = cosine_direction(n2, m.seed, dir_counter(q, M, 1));
    store_pe_split3(X_w, wj);
    bool ok = true;
    for (int j = 0; j < M; ++j) {
      ok = irt_layer1();
      if (!ok) break;
      const f3 c = env_lookup(m.env, m.env_h, m.env_w, wj) * brdf_eval(a2, r2, n2, wj, wo2, m.f0, m.lambert);
      wait();
      epilogue_split3(D_w, H_w);
      ok = irt_layer2();
      if (!ok) break;
      if (j + 1 < M) {   // layer 1 is done with X, layer 2 reads H
        wj = cosine_direction(n2, m.seed, dir_counter(q, M, 2 + j));
        store_pe_split3(X_w, wj);
      }
      wait();
      lo2 = lo2 + c * visibility_from_logit(head_vis_s(D_w, hv, sw[OFF_IB3]), m.force_vis2, m.hard);
    }
    if (!ok) break;
    lo2 = lo2 * (kPi / (float)M);

    // Eq. 2 then the primary term of Eq. 1
    const f3 li = env_lookup(m.env, m.env_h, m.env_w, wi) * v + lo2 * (1.0f - v);
    const f3 c = li * (m.mis ? mis_weighted_brdf(m, xyz(ar), ar.w, n, wo, wi)
                             : brdf_eval(xyz(ar), ar.w, n, wi, wo, m.f0, m.lambert));
    red[t] = make_float4(c.x, c.y, c.z, 0.f);
    wg_sync(wg);
    for (int s = warp; s < npix; s += 4) {
      const int ra = max(0, s * N - off0), rb = min(nvalid, (s + 1) * N - off0);
      f3 sum = mk(0.f, 0.f, 0.f);
      if (s == 0 && off0 > 0) {
        const float4 cs = carry[32 * parity + lane];
        sum = mk(cs.x, cs.y, cs.z);
      }
      const int i_a = off0 + ra - s * N;                       // direction of row ra
      for (int r = ra + ((lane - i_a) & 31); r < rb; r += 32) {
        const float4 h = red[r];
        sum = mk(sum.x + h.x, sum.y + h.y, sum.z + h.z);
      }
      if ((s + 1) * N - off0 <= nvalid) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          sum.x += __shfl_xor_sync(0xffffffffu, sum.x, o);
          sum.y += __shfl_xor_sync(0xffffffffu, sum.y, o);
          sum.z += __shfl_xor_sync(0xffffffffu, sum.z, o);
        }
        if (lane == 0) {
          const float sc = kPi / (float)N;
          out[p_first + s] = make_float4(sum.x * sc, sum.y * sc, sum.z * sc, 0.0f);
        }
      } else {
        carry[32 * (parity ^ 1u) + lane] = make_float4(sum.x, sum.y, sum.z, 0.f);
      }
    }
  }

  // ---- teardown: drain, then free TMEM
  abort = wg_sync_or(wg, abort);
  if (abort && t == 0) (void)mbar_wait(bar, pending_phase);   // let an MMA still in flight finish
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(kTmemCols) : "memory");
}

}  // namespace

cudaError_t prepare_render_fp32() {
  const cudaError_t e =
      cudaFuncSetAttribute(render_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  // smallest carveout (percent of the 228 KB maximum) that holds the CTA; the rest of the SM's 256 KB serves as L1
  return cudaFuncSetAttribute(render_fp32_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)(((kSmemBytes + 1024) * 100 + 233471) / 233472));
}

cudaError_t launch_render_fp32(const ModelDesc& m, const rt_gbuffer& gb, int P, long long offset, float4* out,
                               int num_sms, cudaStream_t s) {
  const int need = (int)(((long long)P + kWG - 1) / kWG);
  const int grid = need < num_sms ? need : num_sms;
  render_fp32_kernel<<<grid, kThreads, kSmemBytes, s>>>(m, gb, P, offset, out);
  return cudaGetLastError();
}

}  // namespace rtk
