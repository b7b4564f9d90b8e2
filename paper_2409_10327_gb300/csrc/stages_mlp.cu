// Stages (b) and (c) on their own: B at given features (rt_decode) and I at
// given features and directions (rt_trace).
// Rows, (point) or (point, direction) consecutively, run 128 at a time through
// the tensor-core layers of tc_split.cuh, as in the FP32 frame kernel: a
// warpgroup per tile, thread = row = TMEM lane, three warpgroups per SM that
// take turns on the tensor pipe.  Within a warpgroup the next tile's features
// and encoding are made while layer 2 of the current one runs.
// A tile is 49 MMAs of 32 cycles against about 1,000 instructions per warp and
// waits on its chains and TMEM reads, hence as many warpgroups as tensor memory
// holds: 160 columns each, the hidden operand taking the input's columns (two
// of 256 columns: 169 us for the trace below).
// 100,003 points with 16 directions: rt_encode + rt_decode + rt_trace took
// 1,184 us with a warp per 32 directions of a point (half of the lanes idle at
// 16) and a thread per decoded point; now 209 us.
#include "tc_split.cuh"

namespace rtk {

namespace {

constexpr int kWG = 3;
constexpr int kThreads = 128 * kWG;
constexpr int kTmemCols = 512;   // 160 per warpgroup; allocations are powers of two
constexpr int TM_D = 0, TM_X = 64, TM_H = TM_X;   // H takes X's columns once layer 1 has read them
// shared memory: one MLP's split weights and output layers, then per warpgroup the tile's split features and a barrier
constexpr int SM_W1 = 0, SM_W2 = 3 * kPart, SM_B2 = 6 * kPart, SM_ONES = SM_B2 + 2048, SM_HEAD = SM_ONES + 4096;
constexpr int SM_WG = SM_HEAD + HD_FLOATS * 4;
constexpr int kSlot = 3 * 64;
constexpr int WG_BAR = kPixSlots * kSlot;
constexpr int WG_BYTES = WG_BAR + 16;
constexpr int kTmemSlot = SM_WG + kWG * WG_BYTES;
constexpr size_t kSmemBytes = kTmemSlot + 16 + 1024;
static_assert(SM_WG % 16 == 0 && WG_BYTES % 16 == 0, "aligned blocks");

// two features of a point's row (k even; zero beyond lf)
__device__ __forceinline__ float2 feat_pair(const float* __restrict__ f, int k, int lf) {
  return k < lf ? make_float2(__ldg(f + k), __ldg(f + k + 1)) : make_float2(0.f, 0.f);
}

// IRT: I on [feat[p] | PE(dirs[p * K + k])] -> vis, depth; otherwise B on feat[p] -> brdf (K = 1).
template <bool IRT>
__global__ void __launch_bounds__(kThreads, 1)
mlp_rows_kernel(const __grid_constant__ ModelDesc m, const float* __restrict__ feat, const float4* __restrict__ dirs,
                long long rows, int K, float* __restrict__ vis, float* __restrict__ depth,
                float4* __restrict__ brdf) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x;
  const int wg = __shfl_sync(0xffffffffu, tid >> 7, 0), t = tid & 127, warp = __shfl_sync(0xffffffffu, t >> 5, 0);
  uint8_t* slots = sm + SM_WG + wg * WG_BYTES;
  const float* hd = reinterpret_cast<const float*>(sm + SM_HEAD);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kTmemSlot);
  const uint32_t bar = smem_u32(slots + WG_BAR);
  if (IRT) {
    build_split_matrix(sm + SM_W1, m.wpack + OFF_IW1F, 32 + kPE, m.wpack + OFF_IB1, tid, kThreads);
    build_split_matrix(sm + SM_W2, m.wpack + OFF_IW2, 64, nullptr, tid, kThreads);
    build_split_bias(sm + SM_B2, m.wpack + OFF_IB2, tid, kThreads);
  } else {
    build_split_matrix(sm + SM_W1, m.wpack + OFF_BW1, 32, m.wpack + OFF_BB1, tid, kThreads);
    build_split_matrix(sm + SM_W2, m.wpack + OFF_BW2, 64, nullptr, tid, kThreads);
    build_split_bias(sm + SM_B2, m.wpack + OFF_BB2, tid, kThreads);
  }
  build_split_ones(sm + SM_ONES, tid, kThreads);
  build_heads(reinterpret_cast<float*>(sm + SM_HEAD), m.wpack, tid, kThreads);
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
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0) + (uint32_t)(160 * wg);
  const uint32_t D_t = tmem + TM_D, X_t = tmem + TM_X, H_t = tmem + TM_H;
  const uint32_t lane_off = (uint32_t)(32 * warp) << 16;
  const uint32_t D_w = D_t + lane_off, X_w = X_t + lane_off, H_w = H_t + lane_off;
  const uint32_t S = smem_u32(sm);
  const int lf = m.lf;

  uint32_t phase = 0, pending_phase = 0;
  int abort = 0;
  // issue / wait as in render_fp32.cu: an abort vote at each issue keeps the warpgroup together
  auto issue = [&](auto chain) -> bool {
    tmem_st_wait();
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
      if (!abort && t == 0) atomicOr(m.status, kStatusTimeout | kWhereStageMlp);
      abort = 1;
      pending_phase = phase;
    }
    phase ^= 1u;
    tc_fence_after();
  };

  // The split layer-1 input of a tile's rows: features through shared memory (split once per point) where the tile
  // spans few points, else per row when they are stored; the encoding in registers.
  uint32_t pe0[16], pe1[16], pe2[16];
  auto prepare_tile = [&](long long tile) {
    const long long r0 = tile * 128, r1 = min(r0 + 128, rows) - 1;
    const long long p0 = r0 / K;
    const int np = (int)(r1 / K - p0) + 1;
    wg_sync(wg);   // the previous tile's slots are read
    if (np <= kPixSlots) {
      for (int e = t; e < np * 16; e += 128) {
        const float2 f = feat_pair(feat + (size_t)(p0 + (e >> 4)) * lf, 2 * (e & 15), lf);
        uint32_t q0, q1, q2;
        split3(f.x, f.y, q0, q1, q2);
        uint32_t* d = reinterpret_cast<uint32_t*>(slots + (e >> 4) * kSlot) + (e & 15);
        d[0] = q0;
        d[16] = q1;
        d[32] = q2;
      }
    }
    // B reads the ones columns only: its weights are zero on the encoding's
    pe_split3(IRT ? xyz(__ldg(dirs + min(r0 + t, r1))) : mk(0.f, 0.f, 0.f), pe0, pe1, pe2);
    wg_sync(wg);
  };
  auto store_input = [&](long long tile) {
    const long long r0 = tile * 128, r1 = min(r0 + 128, rows) - 1;
    const long long p0 = r0 / K, p = min(r0 + t, r1) / K;
    tmem_st16x3(X_w + 16, pe0, pe1, pe2);
    if ((int)(r1 / K - p0) + 1 <= kPixSlots) {
      const uint8_t* src = slots + (int)(p - p0) * kSlot;
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        uint32_t fr[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint4 v = *reinterpret_cast<const uint4*>(src + part * 64 + 16 * c);
          fr[4 * c] = v.x;
          fr[4 * c + 1] = v.y;
          fr[4 * c + 2] = v.z;
          fr[4 * c + 3] = v.w;
        }
        tmem_st16(X_w + 32 * part, fr);
      }
    } else {
      uint32_t q0[16], q1[16], q2[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        const float2 f = feat_pair(feat + (size_t)p * lf, 2 * e, lf);
        split3(f.x, f.y, q0[e], q1[e], q2[e]);
      }
      tmem_st16x3(X_w, q0, q1, q2);
    }
  };

  const long long ntiles = (rows + 127) / 128;
  const long long stride = (long long)gridDim.x * kWG;
  long long tile = (long long)blockIdx.x * kWG + wg;
  if (tile < ntiles) {
    prepare_tile(tile);
    store_input(tile);
  }
  for (; tile < ntiles; tile += stride) {
    if (!issue([&](uint32_t one) {
          if (IRT) mma_split3<0, 4>(one, D_t, X_t, S + SM_W1);
          else mma_split3_brdf1(one, D_t, X_t, S + SM_W1);
        }))
      break;
    wait();
    epilogue_split3(D_w, H_w);
    if (!issue([&](uint32_t one) { mma_split3_layer2(one, D_t, H_t, S + SM_W2, S + SM_ONES, S + SM_B2); })) break;
    if (tile + stride < ntiles) prepare_tile(tile + stride);
    wait();
    if (tile + stride < ntiles) store_input(tile + stride);
    const long long r = tile * 128 + t;
    if (IRT) {
      float z[2];
      head_fp32<2, 2>(D_w, hd + HD_IW3, hd + HD_IB3, z);
      if (r < rows) {
        vis[r] = sigmoidf_(z[0]);
        depth[r] = depth_from_logit(z[1], m.near_t, m.far_t);
      }
    } else {
      float y[7];
      head_fp32<7, 8>(D_w, hd + HD_BW3, hd + HD_BB3, y);
      if (r < rows) {
        const float inv = rsqrtf(fmaxf(y[0] * y[0] + y[1] * y[1] + y[2] * y[2], 1e-24f));
        brdf[2 * r] = make_float4(y[0] * inv, y[1] * inv, y[2] * inv, sigmoidf_(y[3]));
        brdf[2 * r + 1] = make_float4(sigmoidf_(y[4]), sigmoidf_(y[5]), 0.09f + 0.91f * sigmoidf_(y[6]), 0.0f);
      }
    }
  }

  abort = wg_sync_or(wg, abort);
  if (abort && t == 0) (void)mbar_wait(bar, pending_phase);   // let an MMA still in flight finish
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*tslot), "r"(kTmemCols) : "memory");
}

template <bool IRT>
cudaError_t prepare_rows() {
  const cudaError_t e =
      cudaFuncSetAttribute(mlp_rows_kernel<IRT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(mlp_rows_kernel<IRT>, cudaFuncAttributePreferredSharedMemoryCarveout,
                              (int)(((kSmemBytes + 1024) * 100 + 233471) / 233472));
}

template <bool IRT>
cudaError_t launch_rows(const ModelDesc& m, const float* feat, const float4* dirs, long long rows, int K, float* vis,
                        float* depth, float4* brdf, int num_sms, cudaStream_t s) {
  const long long need = ((rows + 127) / 128 + kWG - 1) / kWG;
  const int grid = (int)(need < num_sms ? need : num_sms);
  mlp_rows_kernel<IRT><<<grid, kThreads, kSmemBytes, s>>>(m, feat, dirs, rows, K, vis, depth, brdf);
  return cudaGetLastError();
}

}  // namespace

cudaError_t prepare_stages_mlp() {
  const cudaError_t e = prepare_rows<true>();
  return e != cudaSuccess ? e : prepare_rows<false>();
}

cudaError_t launch_decode(const ModelDesc& m, const float* feat, int P, float* brdf, int num_sms, cudaStream_t s) {
  return launch_rows<false>(m, feat, nullptr, P, 1, nullptr, nullptr, reinterpret_cast<float4*>(brdf), num_sms, s);
}

cudaError_t launch_trace(const ModelDesc& m, const float* feat, const float4* dirs, int P, int K, float* vis,
                         float* depth, int num_sms, cudaStream_t s) {
  return launch_rows<true>(m, feat, dirs, (long long)P * K, K, vis, depth, nullptr, num_sms, s);
}

}  // namespace rtk
