// Shared pieces of the hand-written FP32 adjoints (rt_backward, rt_distill_backward):
// the warp-level adjoints of the MLP layers (32 rows per warp, activations in
// the k-major layout of warp_gemm.cuh), the accumulators of I's weight
// gradients, the adjoint of the trilinear hash encode, and the flush of the
// accumulators into the caller's gradient blob.
//
// I runs 1 + M times per row chunk (B once), so its layers are all register
// tiles: the forward and the transposed products (dZ1 = dZ2 W2, against a
// transposed copy of W2 in shared memory) are 32 x 64 warp GEMMs, and a weight
// gradient is a 64 x 64 (64 x 32) outer product over the warp's 32 rows with
// 64 outputs per lane.  Its sum over the whole launch lives in tensor memory,
// used as 256 words of private storage per lane (8 warps, two per TMEM lane
// quarter): a chunk's 64 x 64 contribution is summed in registers and added
// to the warp's accumulator by one tcgen05.ld / st of the lane's 64 words.
// (A shared-memory accumulator per CTA took 246 float atomics per lane and
// evaluation, more time than the products.)  B adds its gradients straight
// into the caller's blob with coalesced global reductions (BlobB).
// Bound by FMA chains and their shared-memory reads at two warps per
// scheduler.  16,384 rays x 64 directions: 13.7 ms, about 30 ms with the
// thread-per-row products and shared atomics; the distillation's kernel on
// 2,048 points x 1,024 directions 0.98 ms, 4.5 ms before.
#pragma once

#include "tc_common.cuh"
#include "warp_gemm.cuh"

namespace rtk {

// Shared-memory weights of an adjoint: I's part of the packed image, then W2 transposed, [out c][in k]
constexpr int OFF_IW2T = OFF_BW1;
constexpr int WADJ_FLOATS = OFF_IW2T + 64 * 64;
static_assert(OFF_IW2T % 4 == 0, "float4 alignment");

constexpr int kAdjWarps = 8;               // warps per CTA, one CTA per SM
constexpr int kAdjThreads = 32 * kAdjWarps;
// TMEM words of a lane
constexpr int TA_W2 = 0;                   // dW2, two passes of 64
constexpr int TA_W1P = 128;                // dW1, PE columns
constexpr int TA_S = 192;                  // backward: the chunk's sum over j of dZ1

__device__ __forceinline__ void load_adjoint_weights(float* sw, const float* __restrict__ wpack) {
  for (int i = threadIdx.x; i < OFF_BW1 / 4; i += kAdjThreads)
    reinterpret_cast<float4*>(sw)[i] = __ldg(reinterpret_cast<const float4*>(wpack) + i);
  for (int i = threadIdx.x; i < 4096; i += kAdjThreads)
    sw[OFF_IW2T + i] = __ldg(wpack + OFF_IW2 + (i & 63) * 64 + (i >> 6));
}

// B's gradient blob (canonical layout of rt_param_count: W1 [64][lf], b1, W2 [64][64], b2, W3 [7][64], b3)
struct BlobB {
  float* g;
  int lf;
  __device__ __forceinline__ float* w1() const { return g; }
  __device__ __forceinline__ float* b1() const { return g + 64 * lf; }
  __device__ __forceinline__ float* w2() const { return g + 64 * lf + 64; }
  __device__ __forceinline__ float* b2() const { return g + 64 * lf + 64 + 4096; }
  __device__ __forceinline__ float* w3() const { return g + 64 * lf + 128 + 4096; }
  __device__ __forceinline__ float* b3() const { return g + 64 * lf + 128 + 4096 + 448; }
};

// ---- tensor memory as per-lane accumulators --------------------------------
__device__ __forceinline__ uint32_t adj_tmem_alloc(uint32_t* slot, int tid) {
  if (tid < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // warp w owns its 32 lanes (w % 4) and columns 256 (w / 4) ..
  return *slot + ((uint32_t)(32 * ((tid >> 5) & 3)) << 16) + (uint32_t)(256 * (tid >> 7));
}
// called by all threads after their last TMEM access
__device__ __forceinline__ void adj_tmem_free(const uint32_t* slot, int tid) {
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid < 32)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*slot), "r"(512) : "memory");
}
// words [0, 16 * n16) of this lane <- 0
__device__ __forceinline__ void tmem_zero(uint32_t taddr, int n16) {
  uint32_t z[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) z[i] = 0u;
  for (int i = 0; i < n16; ++i) tmem_st16(taddr + 16 * i, z);
  tmem_st_wait();
}
// 64 words of this lane += v
__device__ __forceinline__ void tmem_add64(uint32_t taddr, const float (&v)[64]) {
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    uint32_t r[16];
    tmem_ld16(taddr + 16 * h, r);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(__uint_as_float(r[i]) + v[16 * h + i]);
    tmem_st16(taddr + 16 * h, r);
  }
  tmem_st_wait();
}
// the same for a Tile (words in v[q][c].x, .y order)
__device__ __forceinline__ void tmem_add_tile(uint32_t taddr, const Tile& t) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t r[16];
    tmem_ld16(taddr + 16 * q, r);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      r[2 * c] = __float_as_uint(__uint_as_float(r[2 * c]) + t.v[q][c].x);
      r[2 * c + 1] = __float_as_uint(__uint_as_float(r[2 * c + 1]) + t.v[q][c].y);
    }
    tmem_st16(taddr + 16 * q, r);
  }
  tmem_st_wait();
}
__device__ __forceinline__ void tmem_load_tile(uint32_t taddr, Tile& t) {
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    uint32_t r[16];
    tmem_ld16(taddr + 16 * q, r);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 8; ++c) t.v[q][c] = make_float2(__uint_as_float(r[2 * c]), __uint_as_float(r[2 * c + 1]));
  }
}

// ---- I's layers -------------------------------------------------------------
// Columns (hidden units) of a lane where it owns two whole columns: the 8 lanes
// of a quarter warp differ in c >> 3, so their float4 row reads hit distinct banks.
__device__ __forceinline__ int own_col(int lane, int kk) { return 8 * (lane & 7) + (lane >> 3) + 4 * kk; }

// Output layer: dZ2(c, row) = (sum_o dz[o][row] W3[c][o]) * [H2(c, row) > 0] over H2 in place, and for the lane's
// two columns gw[kk][o] += sum_rows H2 dz[o], gb[kk] += sum_rows dZ2.  W3 is [64][2].
template <int NOUT>
__device__ __forceinline__ void bwd_out(float* H2, const float* dz, const float* W3, float (&gw)[2][2], float (&gb)[2],
                                        int lane) {
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const int c = own_col(lane, kk);
    const float w0 = W3[2 * c], w1 = NOUT > 1 ? W3[2 * c + 1] : 0.0f;
    float s0 = 0.f, s1 = 0.f, sb = 0.f;
#pragma unroll
    for (int r = 0; r < 32; r += 4) {
      float4* hp = reinterpret_cast<float4*>(H2 + aidx(c, r));
      const float4 h4 = *hp, z4 = *reinterpret_cast<const float4*>(dz + r);
      const float4 y4 = NOUT > 1 ? *reinterpret_cast<const float4*>(dz + 32 + r) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float h[4] = {h4.x, h4.y, h4.z, h4.w}, z[4] = {z4.x, z4.y, z4.z, z4.w}, y[4] = {y4.x, y4.y, y4.z, y4.w};
      float g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        g[u] = z[u] * w0;
        if (NOUT > 1) g[u] = fmaf(y[u], w1, g[u]);
        g[u] = h[u] > 0.0f ? g[u] : 0.0f;
        sb += g[u];
        s0 = fmaf(h[u], z[u], s0);
        if (NOUT > 1) s1 = fmaf(h[u], y[u], s1);
      }
      *hp = make_float4(g[0], g[1], g[2], g[3]);
    }
    gw[kk][0] += s0;
    if (NOUT > 1) gw[kk][1] += s1;
    gb[kk] += sb;
  }
}

// One outer product over the warp's rows: v[i * NK + j] = sum_rows D(c0 + i, row) A(k0 + j, row), 64 outputs a lane.
template <int NC, int NK>
__device__ __forceinline__ void outer64(const float* A, const float* D, int k0, int c0, float (&v)[64]) {
  static_assert(NC * NK == 64, "64 outputs per lane");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = 0.0f;
#pragma unroll 1
  for (int r = 0; r < 32; r += 4) {
    float4 a[NK];
#pragma unroll
    for (int j = 0; j < NK; ++j) a[j] = *reinterpret_cast<const float4*>(A + aidx(k0 + j, r));
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const float4 d = *reinterpret_cast<const float4*>(D + aidx(c0 + i, r));
#pragma unroll
      for (int j = 0; j < NK; ++j) {
        float s = v[i * NK + j];
        s = fmaf(a[j].x, d.x, s);
        s = fmaf(a[j].y, d.y, s);
        s = fmaf(a[j].z, d.z, s);
        v[i * NK + j] = fmaf(a[j].w, d.w, s);
      }
    }
  }
}
// dW2 += dZ2^T H1 into the warp's accumulator (lane: rows c = 32 pass + 8 rg.., columns k = 8 cg..)
__device__ __forceinline__ void acc_w2(const float* H1, const float* DZ2, uint32_t tacc, int rg, int cg) {
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    float v[64];
    outer64<8, 8>(H1, DZ2, 8 * cg, 32 * pass + 8 * rg, v);
    tmem_add64(tacc + TA_W2 + 64 * pass, v);
  }
}
// dW1's PE columns += dZ1^T PE (lane: rows c = 16 rg.., columns k = 4 cg..)
__device__ __forceinline__ void acc_w1p(const float* PE, const float* DZ1, uint32_t tacc, int rg, int cg) {
  float v[64];
  outer64<16, 4>(PE, DZ1, 4 * cg, 16 * rg, v);
  tmem_add64(tacc + TA_W1P, v);
}

// dZ1 = (dZ2 W2) masked by H1 > 0, over H1 in place (t: the masked tile).  Every lane has read H1 before.
__device__ __forceinline__ void bwd_hidden_tile(const float* DZ2, const float* W2T, float* H1, Tile& t, int rg, int cg) {
  zero(t);
  warp_gemm<kHidden>(DZ2, W2T, t, rg, cg);
  __syncwarp();
  store_masked(H1, t, rg, cg);
  __syncwarp();
}

// sum over the warp's rows of the lane's two columns
__device__ __forceinline__ void col_sums(const float* D, float (&s)[2], int lane) {
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    float a = 0.0f;
#pragma unroll
    for (int r = 0; r < 32; r += 4) {
      const float4 d = *reinterpret_cast<const float4*>(D + aidx(own_col(lane, kk), r));
      a += (d.x + d.y) + (d.z + d.w);
    }
    s[kk] += a;
  }
}

// Where f is shared by the rows (a pixel's or a point's directions), with cs[c] the sum over rows of dZ1:
// dW1f[c][k] += f[k] cs[c] (coalesced global reductions) and, returned in lane k, dLoss/df[k] = sum_c cs[c] W1f[k][c].
__device__ __forceinline__ float bwd_shared_feature(const float* f, const float* cs, const float* W1F, int lf,
                                                    float* __restrict__ g_irt, int lane) {
  float s = 0.0f;
  if (lane < lf) {
    const int in_i = lf + kPE;
    const float fk = f[lane];
#pragma unroll 8
    for (int c = 0; c < 64; ++c) atomicAdd(g_irt + c * in_i + lane, fk * cs[c]);
#pragma unroll 8
    for (int cc = 0; cc < 64; ++cc) {
      const int c = (cc + lane) & 63;   // rotated: the lanes' rows of W1F share banks
      s = fmaf(cs[c], W1F[lane * 64 + c], s);
    }
  }
  return s;
}

// gW[c][k] += sum_rows A(k, row) D(c, row) for c < 64, k < K, rows of gW ld apart: lane = k, so the reductions into
// global memory are coalesced; gb[c] += sum_rows D(c, row) if gb != nullptr.
__device__ __forceinline__ void bwd_weights_global(const float* A, int K, const float* D, float* __restrict__ gW, int ld,
                                                   float* __restrict__ gb, int lane) {
  for (int k0 = 0; k0 < K; k0 += 32) {
    const int k = k0 + lane;
    const bool live = k < K;
    float a[32];
#pragma unroll
    for (int r = 0; r < 32; r += 4) {
      const float4 v = *reinterpret_cast<const float4*>(A + aidx(live ? k : k0, r));
      a[r] = v.x;
      a[r + 1] = v.y;
      a[r + 2] = v.z;
      a[r + 3] = v.w;
    }
    for (int c = 0; c < 64; ++c) {
      float s = 0.0f;
#pragma unroll
      for (int r = 0; r < 32; r += 4) {
        const float4 d = *reinterpret_cast<const float4*>(D + aidx(c, r));
        s = fmaf(a[r], d.x, s);
        s = fmaf(a[r + 1], d.y, s);
        s = fmaf(a[r + 2], d.z, s);
        s = fmaf(a[r + 3], d.w, s);
      }
      if (live) atomicAdd(gW + c * ld + k, s);
    }
  }
  if (gb != nullptr) {
    float s[2] = {0.f, 0.f};
    col_sums(D, s, lane);
    atomicAdd(gb + own_col(lane, 0), s[0]);
    atomicAdd(gb + own_col(lane, 1), s[1]);
  }
}

// ---- B's layers (one evaluation per chunk; weights through the read-only cache) ----
// DZ2(c, row) = (sum_o dz[o][row] W3[c][o]) * [H2(c, row) > 0]   (thread per row)
template <int NOUT, int LDW>
__device__ __forceinline__ void bwd_head(const float* H2, const float* dz, const float* W3, float* DZ2, int lane) {
  float g[NOUT];
#pragma unroll
  for (int o = 0; o < NOUT; ++o) g[o] = dz[o * 32 + lane];
#pragma unroll 8
  for (int c = 0; c < 64; ++c) {
    float s = 0.0f;
#pragma unroll
    for (int o = 0; o < NOUT; ++o) s = fmaf(g[o], __ldg(W3 + c * LDW + o), s);
    DZ2[aidx(c, lane)] = H2[aidx(c, lane)] > 0.0f ? s : 0.0f;
  }
}

// dW3[o][k] += sum_rows H2(k, row) dz[o][row]; db3[o] += sum_rows dz[o][row]
template <int NOUT>
__device__ __forceinline__ void bwd_w3(const float* H2, const float* dz, float* gW3, float* gb3, int lane, int ld) {
#pragma unroll 1   // rolled: unrolled, the two passes' global atomics keep too many registers live
  for (int kk = 0; kk < 2; ++kk) {
    const int k = own_col(lane, kk);
    float acc[NOUT];
#pragma unroll
    for (int o = 0; o < NOUT; ++o) acc[o] = 0.0f;
    for (int r = 0; r < 32; r += 4) {
      const float4 h = *reinterpret_cast<const float4*>(H2 + aidx(k, r));
#pragma unroll
      for (int o = 0; o < NOUT; ++o) {
        const float4 z = *reinterpret_cast<const float4*>(dz + o * 32 + r);
        acc[o] = fmaf(h.w, z.w, fmaf(h.z, z.z, fmaf(h.y, z.y, fmaf(h.x, z.x, acc[o]))));
      }
    }
#pragma unroll
    for (int o = 0; o < NOUT; ++o) atomicAdd(gW3 + o * ld + k, acc[o]);
  }
  if (lane < NOUT) {
    float s = 0.0f;
    for (int r = 0; r < 32; ++r) s += dz[lane * 32 + r];
    atomicAdd(gb3 + lane, s);
  }
}

// OUT(k, row) = (sum_c D(c, row) W[k][c]) * [MASK(k, row) > 0] for k < 64 (thread per row);
// W is a [64][64] matrix in global memory stored [k][c]
__device__ __forceinline__ void bwd_hidden(const float* D, const float* __restrict__ W, const float* MASK, float* OUT,
                                           int lane) {
  float d[64];
#pragma unroll
  for (int c = 0; c < 64; ++c) d[c] = D[aidx(c, lane)];
#pragma unroll 2
  for (int k = 0; k < 64; ++k) {
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < 64; c += 4) {
      const float4 w = __ldg(reinterpret_cast<const float4*>(W + k * 64 + c));
      s = fmaf(d[c], w.x, s);
      s = fmaf(d[c + 1], w.y, s);
      s = fmaf(d[c + 2], w.z, s);
      s = fmaf(d[c + 3], w.w, s);
    }
    OUT[aidx(k, lane)] = MASK[aidx(k, lane)] > 0.0f ? s : 0.0f;
  }
}

// din[k] += sum_c D(c, row) W[k][c] for k < K (thread per row)
__device__ __forceinline__ void bwd_input(const float* D, const float* W, int K, float (&din)[32], int lane) {
  float d[64];
#pragma unroll
  for (int c = 0; c < 64; ++c) d[c] = D[aidx(c, lane)];
#pragma unroll
  for (int k = 0; k < 32; ++k) {
    if (k < K) {
      float s = 0.0f;
#pragma unroll
      for (int c = 0; c < 64; c += 4) {
        const float4 w = *reinterpret_cast<const float4*>(W + k * 64 + c);
        s = fmaf(d[c], w.x, s);
        s = fmaf(d[c + 1], w.y, s);
        s = fmaf(d[c + 2], w.z, s);
        s = fmaf(d[c + 3], w.w, s);
      }
      din[k] += s;
    }
  }
}

// trilinear encode adjoint at point x for one level: table gradient scatter
// and (optionally) dLoss/dx
__device__ __forceinline__ void encode_level_bwd(const GridDesc& g, int l, f3 x, float df0, float df1,
                                                 float* __restrict__ g_table, f3* dx) {
  const int res = g.res[l];
  uint32_t ix, iy, iz;
  float wx, wy, wz;
  grid_cell_exact(x.x, res, ix, wx);
  grid_cell_exact(x.y, res, iy, wy);
  grid_cell_exact(x.z, res, iz, wz);
  const size_t base = (size_t)l << g.log2T;
  const int dense = g.dense[l];
  float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int ox = c & 1, oy = (c >> 1) & 1, oz = (c >> 2) & 1;
    const uint32_t row = corner_row(ix + ox, iy + oy, iz + oz, res, dense, g.mask);
    const float ax = ox ? wx : 1.0f - wx, ay = oy ? wy : 1.0f - wy, az = oz ? wz : 1.0f - wz;
    const float w = ax * ay * az;
    atomicAdd(reinterpret_cast<float2*>(g_table) + base + row, make_float2(w * df0, w * df1));
    if (dx != nullptr) {
      const float2 e = table_entry(g, base + row);
      const float de = e.x * df0 + e.y * df1;
      gx += de * (ox ? 1.0f : -1.0f) * ay * az;
      gy += de * (oy ? 1.0f : -1.0f) * ax * az;
      gz += de * (oz ? 1.0f : -1.0f) * ax * ay;
    }
  }
  if (dx != nullptr) {
    // dg/dx = N_l / 2 inside the box, 0 on a clamped axis
    const float s = 0.5f * (float)res;
    const float ux = x.x * 0.5f + 0.5f, uy = x.y * 0.5f + 0.5f, uz = x.z * 0.5f + 0.5f;
    dx->x += (ux >= 0.0f && ux <= 1.0f) ? gx * s : 0.0f;
    dx->y += (uy >= 0.0f && uy <= 1.0f) ? gy * s : 0.0f;
    dx->z += (uz >= 0.0f && uz <= 1.0f) ? gz * s : 0.0f;
  }
}

// Bitonic sort of one 32-bit key per lane across the warp, ascending with the
// lane index.  All 32 lanes take part.
__device__ __forceinline__ uint32_t warp_sort_u32(uint32_t key) {
  const unsigned lane = threadIdx.x & 31u;
#pragma unroll
  for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      const uint32_t other = __shfl_xor_sync(0xffffffffu, key, j);
      const bool up = (lane & (unsigned)k) == 0u;     // this k-block is sorted ascending
      const bool lower = (lane & (unsigned)j) == 0u;  // this lane is the lower position of its pair
      key = (lower == up) ? min(key, other) : max(key, other);
    }
  }
  return key;
}
// An integer of up to 10 bits spread to every third bit (the Morton interleave of one axis).
__device__ __forceinline__ uint32_t morton_spread(uint32_t v) {
  v &= 0x3FFu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}
// The cell of coordinate u in [-1, 1] on a 256-cell axis (clamped).
__device__ __forceinline__ uint32_t morton_cell8(float u) {
  const float q = fminf(fmaxf((u * 0.5f + 0.5f) * 256.0f, 0.0f), 255.0f);
  return (uint32_t)q;
}

// The encode adjoint at the warp's 32 points (one per lane; `valid` marks the
// real ones): for every level, the table
// gradient of the 8 corners of each point's cell and dLoss/dx.  df holds the
// lane's dLoss/df as FP32 bits, features (2l, 2l + 1) of level l.
// Segmented scatter: the warp's points are first put in Morton order of their
// position (8 bits per axis) by a bitonic sort across the lanes, so that points
// that share a table row on a level sit, for the most part, in consecutive
// lanes.  Each run of consecutive lanes on one row is summed by a shuffle tree
// bounded by the run (a fixed order of additions) and reaches the table as one
// float2 reduction; a row whose points are not consecutive receives one
// reduction per run.  Levels without runs cost one ballot per corner over the
// plain scatter.  With WANT_DX, returns dLoss/dx of this lane's own point, and
// scratch is 512 bytes of the warp's shared memory (the points' dx on their way
// back); without it, returns zero and scratch is unused (may be null).
template <bool WANT_DX = true>
__device__ __forceinline__ f3 encode_bwd_sorted(const GridDesc& g, f3 x, const uint32_t (&df)[32], bool valid,
                                                float* __restrict__ g_table, float4* scratch) {
  const unsigned lane = threadIdx.x & 31u;
  const uint32_t code = (morton_spread(morton_cell8(x.x)) << 2) | (morton_spread(morton_cell8(x.y)) << 1) |
                        morton_spread(morton_cell8(x.z));   // 24 bits
  // key: invalid flag, Morton code, lane (unique, so the sort is a permutation of the lanes)
  const uint32_t key = warp_sort_u32((valid ? 0u : 0x80000000u) | (code << 5) | lane);
  const int src = (int)(key & 31u);
  const int nv = __popc(__ballot_sync(0xffffffffu, valid));
  const bool live = (int)lane < nv;   // the valid points come first in the sorted order
  const f3 xs = mk(__shfl_sync(0xffffffffu, x.x, src), __shfl_sync(0xffffffffu, x.y, src),
                   __shfl_sync(0xffffffffu, x.z, src));
  uint32_t d[32];
#pragma unroll
  for (int k = 0; k < 32; ++k) d[k] = __shfl_sync(0xffffffffu, df[k], src);

  f3 dx = mk(0.f, 0.f, 0.f);
#pragma unroll 1
  for (int l = 0; l < g.levels; ++l) {
    float df0 = 0.f, df1 = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (k == l) {
        df0 = __uint_as_float(d[2 * k]);
        df1 = __uint_as_float(d[2 * k + 1]);
      }
    const int res = g.res[l];
    uint32_t ix, iy, iz;
    float wx, wy, wz;
    grid_cell_exact(xs.x, res, ix, wx);
    grid_cell_exact(xs.y, res, iy, wy);
    grid_cell_exact(xs.z, res, iz, wz);
    const size_t base = (size_t)l << g.log2T;
    const int dense = g.dense[l];
    float gx = 0.f, gy = 0.f, gz = 0.f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int ox = c & 1, oy = (c >> 1) & 1, oz = (c >> 2) & 1;
      const uint32_t row = corner_row(ix + ox, iy + oy, iz + oz, res, dense, g.mask);
      const float ax = ox ? wx : 1.0f - wx, ay = oy ? wy : 1.0f - wy, az = oz ? wz : 1.0f - wz;
      const float w = ax * ay * az;
      float v0 = w * df0, v1 = w * df1;
      const uint32_t prev = __shfl_up_sync(0xffffffffu, row, 1);
      const bool head = lane == 0u || prev != row || !live;
      const unsigned heads = __ballot_sync(0xffffffffu, head);
      if (heads != 0xffffffffu) {
        // this lane's run is [lane, end): end is the next head (32 if none)
        const unsigned rest = heads & ~((2u << lane) - 1u);
        const unsigned end = rest ? (unsigned)(__ffs(rest) - 1) : 32u;
        const unsigned span = __reduce_max_sync(0xffffffffu, head ? end - lane : 0u);
        for (unsigned s = 1; s < span; s <<= 1) {
          const float o0 = __shfl_down_sync(0xffffffffu, v0, s);
          const float o1 = __shfl_down_sync(0xffffffffu, v1, s);
          if (lane + s < end) {
            v0 += o0;
            v1 += o1;
          }
        }
      }
      if (head && live) atomicAdd(reinterpret_cast<float2*>(g_table) + base + row, make_float2(v0, v1));
      if (WANT_DX && live) {
        const float2 e = table_entry(g, base + row);
        const float de = e.x * df0 + e.y * df1;
        gx += de * (ox ? 1.0f : -1.0f) * ay * az;
        gy += de * (oy ? 1.0f : -1.0f) * ax * az;
        gz += de * (oz ? 1.0f : -1.0f) * ax * ay;
      }
    }
    if (WANT_DX) {
      // dg/dx = N_l / 2 inside the box, 0 on a clamped axis
      const float s = 0.5f * (float)res;
      const float ux = xs.x * 0.5f + 0.5f, uy = xs.y * 0.5f + 0.5f, uz = xs.z * 0.5f + 0.5f;
      dx.x += (ux >= 0.0f && ux <= 1.0f) ? gx * s : 0.0f;
      dx.y += (uy >= 0.0f && uy <= 1.0f) ? gy * s : 0.0f;
      dx.z += (uz >= 0.0f && uz <= 1.0f) ? gz * s : 0.0f;
    }
  }
  if (!WANT_DX) return dx;
  // back to the lane that owns the point
  scratch[src] = make_float4(dx.x, dx.y, dx.z, 0.0f);
  __syncwarp();
  const float4 r = scratch[lane];
  __syncwarp();
  return mk(r.x, r.y, r.z);
}

// s = D F Vis of the simplified Disney model and its derivatives with respect
// to the roughness r and the normal n (w_i, w_o fixed).  The n-derivative is
// the textbook one (n.h, n.w_i, n.w_o as independent inputs); the component
// along n is irrelevant because the decoder's normal is normalised.
__device__ __forceinline__ float spec_with_grad(float rough, f3 n, f3 wi, f3 wo, float f0, float& ds_dr, f3& ds_dn) {
  const float alpha = rough * rough;
  const float a2 = alpha * alpha;
  const float ndl = dot(n, wi), ndv = dot(n, wo);
  const float nol = fmaxf(ndl, 0.0f), nov = fmaxf(ndv, 1e-4f);
  const f3 hv = wi + wo;
  const float hl2 = dot(hv, hv);
  f3 h = mk(0.f, 0.f, 0.f);
  float ndh = 0.0f, voh = 0.0f, q = 1.0f;
  if (hl2 > 1e-20f) {
    const float inv = rsqrtf(hl2);
    h = hv * inv;
    ndh = dot(n, h);
    voh = 0.5f * hl2 * inv;
    if (ndh > 0.0f) {
      const f3 c = cross(n, h);
      q = dot(c, c) + ndh * ndh * a2;     // = (n.h)^2 (a2 - 1) + 1 on the unit sphere
    }
  }
  const float noh = fmaxf(ndh, 0.0f);
  const float D = a2 / (kPi * q * q);
  const float om = 1.0f - voh;
  const float om2 = om * om;
  const float F = f0 + (1.0f - f0) * (om2 * om2 * om);
  const float A = sqrtf(nov * nov * (1.0f - a2) + a2);
  const float B = sqrtf(nol * nol * (1.0f - a2) + a2);
  const float den = nol * A + nov * B;
  const float vis = 0.5f / den;
  const float dD_da2 = 1.0f / (kPi * q * q) - 2.0f * a2 * noh * noh / (kPi * q * q * q);
  const float dD_dnoh = -4.0f * a2 * noh * (a2 - 1.0f) / (kPi * q * q * q);
  const float dvis_dden = -0.5f / (den * den);
  const float dden_da2 = nol * (1.0f - nov * nov) / (2.0f * A) + nov * (1.0f - nol * nol) / (2.0f * B);
  const float dden_dnol = A + nov * nol * (1.0f - a2) / B;
  const float dden_dnov = nol * nov * (1.0f - a2) / A + B;
  const float ds_da2 = F * (dD_da2 * vis + D * dvis_dden * dden_da2);
  ds_dr = ds_da2 * 4.0f * rough * rough * rough;
  const float g_nol = ndl > 0.0f ? F * D * dvis_dden * dden_dnol : 0.0f;
  const float g_nov = ndv > 1e-4f ? F * D * dvis_dden * dden_dnov : 0.0f;
  const float g_noh = ndh > 0.0f ? F * vis * dD_dnoh : 0.0f;
  ds_dn = wi * g_nol + wo * g_nov + h * g_noh;
  return D * F * vis;
}

// ---- I's weight gradients to the caller -------------------------------------
// The gradients a lane keeps in registers: for its two columns dW3, db2 and db1, and its rows' db3.
struct IrtGrads {
  float w3[2][2], b2[2], b1[2], b3[2];
};
__device__ __forceinline__ void zero(IrtGrads& g) {
#pragma unroll
  for (int i = 0; i < 2; ++i) g.w3[i][0] = g.w3[i][1] = g.b2[i] = g.b1[i] = g.b3[i] = 0.0f;
}

// Sum the warps' accumulators over the CTA in shared memory (buf: kAdjWarps blocks of 4160 floats, `stride` floats
// apart) and add them to the caller's blob (canonical layout of rt_param_count), coalesced.  All threads call it.
__device__ __forceinline__ void flush_irt_grads(float* buf, int stride, uint32_t tacc, IrtGrads& g, int lf,
                                                float* __restrict__ g_irt) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, rg = lane >> 3, cg = lane & 7;
  const int in_i = lf + kPE;
  const int iB1 = 64 * in_i, iW2 = iB1 + 64, iB2 = iW2 + 4096, iW3 = iB2 + 64, iB3 = iW3 + 128;
  float* mine = buf + warp * stride;
  auto cta_sum = [&](int e) {
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < kAdjWarps; ++w) s += buf[w * stride + e];
    return s;
  };
  __syncthreads();
#pragma unroll 1
  for (int part = 0; part < 3; ++part) {   // the two halves of dW2, then dW1's PE columns
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      uint32_t r[16];
      tmem_ld16(tacc + 64 * part + 16 * h, r);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i += 4) {
        const int e = 16 * h + i;
        // parts 0, 1: [32 rows][64]; part 2: [64 rows][32]
        const int o = part < 2 ? (8 * rg + (e >> 3)) * 64 + 8 * cg + (e & 7) : (16 * rg + (e >> 2)) * 32 + 4 * cg;
        *reinterpret_cast<float4*>(mine + o) = make_float4(__uint_as_float(r[i]), __uint_as_float(r[i + 1]),
                                                           __uint_as_float(r[i + 2]), __uint_as_float(r[i + 3]));
      }
    }
    __syncthreads();
    for (int e = tid; e < 2048; e += kAdjThreads) {
      if (part < 2) atomicAdd(g_irt + iW2 + 2048 * part + e, cta_sum(e));
      else if ((e & 31) < kPE) atomicAdd(g_irt + (e >> 5) * in_i + lf + (e & 31), cta_sum(e));
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    g.b3[0] += __shfl_xor_sync(0xffffffffu, g.b3[0], o);
    g.b3[1] += __shfl_xor_sync(0xffffffffu, g.b3[1], o);
  }
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const int c = own_col(lane, kk);
    mine[c] = g.w3[kk][0];
    mine[64 + c] = g.w3[kk][1];
    mine[128 + c] = g.b2[kk];
    mine[192 + c] = g.b1[kk];
  }
  if (lane < 2) mine[256 + lane] = g.b3[lane];
  __syncthreads();
  for (int e = tid; e < 258; e += kAdjThreads) {
    const int o = e < 128 ? iW3 + e : e < 192 ? iB2 + e - 128 : e < 256 ? iB1 + e - 192 : iB3 + e - 256;
    atomicAdd(g_irt + o, cta_sum(e));
  }
}

}  // namespace rtk
