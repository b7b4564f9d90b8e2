// FP32 MLP layers on the bf16 tensor cores: every operand is carried as three
// bf16 parts (a = a0 + a1 + a2 exactly, 8 significant bits each), and a
// product keeps the six partial products down to 2^-18 of the largest,
//   a2 w0 + a1 w1 + a0 w2 + a1 w0 + a0 w1 + a0 w0   (smallest first),
// accumulated in FP32 in tensor memory.  The dropped ones are below 2^-25 of
// |a w|, under the rounding of an FP32 product; a 64-term layer rounds 4
// times at full magnitude here against 64 times in an FFMA chain.  Measured
// against 64-bit sums the error is no larger than the chains': 3.4e-5 for both
// over the stage calls' outputs, and 2.6e-5 to 8.5e-4 against 3.6e-5 to 8.9e-4
// for whole frames.  The bf16 range is FP32's, so no scaling is needed.  Parts
// 0 and 1 saturate, so that an infinite operand does not turn the residuals
// into NaN; its part 2, the rest, is infinite, and so are its products.
//
// Conventions as in tc_common.cuh (a warpgroup owns 128 TMEM lanes, thread t =
// row t); a split operand in TMEM is three blocks of 32 columns.
#pragma once

#include "mbarrier.cuh"
#include "tc_common.cuh"

namespace rtk {

// Split weights in shared memory: per 64 x 64 matrix three K-major tiles (parts
// 0, 1, 2), 128-byte swizzle, 1024-byte aligned.  Layer-1 biases ride on the
// ones columns kBiasCol .. kBiasCol + 2 (the three parts of b1, in part 0 of
// the tile); layer-2 biases on a ones tile times a K = 16 bias tile holding the
// three parts of b2.
constexpr int kPart = 8192;
// FP32 output layers (floats)
constexpr int HD_IW3 = 0;                    // [64][2]
constexpr int HD_BW3 = HD_IW3 + 128;         // [64][8]
constexpr int HD_IB3 = HD_BW3 + 512;         // [4]
constexpr int HD_BB3 = HD_IB3 + 4;           // [8]
constexpr int HD_FLOATS = HD_BB3 + 8;

// bf16 pair, rounded; an infinite value becomes the largest finite one
__device__ __forceinline__ uint32_t pack_bf16_sat(float lo, float hi) {
  uint32_t d;
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(hi), "f"(lo));
  return d;
}
// The three bf16 parts of a pair: q0 and q1 rounded, q2 the exact rest (its
// high halves: at most 8 significant bits are left).
__device__ __forceinline__ void split3(float a, float b, uint32_t& q0, uint32_t& q1, uint32_t& q2) {
  q0 = pack_bf16_sat(a, b);
  float2 r = __fadd2_rn(make_float2(a, b), make_float2(-bf16_lo_half(q0), -bf16_hi_half(q0)));
  q1 = pack_bf16_sat(r.x, r.y);
  r = __fadd2_rn(r, make_float2(-bf16_lo_half(q1), -bf16_hi_half(q1)));
  q2 = __byte_perm(__float_as_uint(r.x), __float_as_uint(r.y), 0x7632);
}

// One 64 x 64 weight matrix as three swizzled tiles from the packed FP32 image:
// element (n, k) is w[k * 64 + n] for k < rows, and b[n]'s parts sit at
// k = kBiasCol .. + 2 of part 0 when b is given.  One thread makes 8 inputs of
// one output, so global reads are coalesced over n and the 16-byte stores of a
// quarter warp hit distinct banks.
__device__ __forceinline__ void build_split_matrix(uint8_t* dst, const float* __restrict__ w, int rows,
                                                   const float* __restrict__ b, int tid, int nthreads) {
  for (int e = tid; e < 64 * 8; e += nthreads) {
    const int n = e & 63, kc = e >> 6;
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * kc + i;
      v[i] = k < rows ? __ldg(w + k * 64 + n) : 0.0f;
    }
    uint32_t q[3][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) split3(v[2 * i], v[2 * i + 1], q[0][i], q[1][i], q[2][i]);
    static_assert(kBiasCol == 59, "bias parts at inputs 59, 60, 61");
    if (b != nullptr && kc == 7) {
      uint32_t p0, p1, p2;
      split3(__ldg(b + n), 0.0f, p0, p1, p2);
      q[0][1] = (q[0][1] & 0xFFFFu) | (p0 << 16);            // inputs 58 | 59
      q[0][2] = (p1 & 0xFFFFu) | (p2 << 16);                 // inputs 60 | 61
    }
#pragma unroll
    for (int p = 0; p < 3; ++p)
      *reinterpret_cast<uint4*>(dst + p * kPart + swz128(n, 8 * kc)) = make_uint4(q[p][0], q[p][1], q[p][2], q[p][3]);
  }
}
// Layer-2 bias tile: row n holds the parts of b[n] and zeros (A is all ones, so the swizzle's order does not matter).
__device__ __forceinline__ void build_split_bias(uint8_t* dst, const float* __restrict__ b, int tid, int nthreads) {
  for (int n = tid; n < 64; n += nthreads) {
    uint32_t p0, p1, p2;
    split3(__ldg(b + n), 0.0f, p0, p1, p2);
    uint4* row = reinterpret_cast<uint4*>(dst + 32 * n);
    row[0] = make_uint4((p0 & 0xFFFFu) | (p1 << 16), p2 & 0xFFFFu, 0u, 0u);
    row[1] = make_uint4(0u, 0u, 0u, 0u);
  }
}
__device__ __forceinline__ void build_split_ones(uint8_t* dst, int tid, int nthreads) {
  for (int i = tid; i < 4096 / 16; i += nthreads)
    reinterpret_cast<uint4*>(dst)[i] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
}
// FP32 output layers of both MLPs.
__device__ __forceinline__ void build_heads(float* hd, const float* __restrict__ wpack, int tid, int nthreads) {
  for (int i = tid; i < 128; i += nthreads) hd[HD_IW3 + i] = __ldg(wpack + OFF_IW3 + i);
  for (int i = tid; i < 512; i += nthreads) hd[HD_BW3 + i] = __ldg(wpack + OFF_BW3 + i);
  for (int i = tid; i < 4; i += nthreads) hd[HD_IB3 + i] = __ldg(wpack + OFF_IB3 + i);
  for (int i = tid; i < 8; i += nthreads) hd[HD_BB3 + i] = __ldg(wpack + OFF_BB3 + i);
}
// The layer-1 tile of I takes [f (32) | PE (32)]: the feature and PE rows of the packed image are adjacent.
static_assert(OFF_IW1P == OFF_IW1F + 32 * 64, "I's layer 1 is one [64][64] block");

template <int K0, int K1>
__device__ __forceinline__ void mma_part(uint32_t one, uint32_t d, uint32_t a_t, uint32_t w_s, uint32_t first) {
#pragma unroll
  for (int k = K0; k < K1; ++k) mma_bf16_ts(one, d, a_t + 8 * k, sdesc(w_s + 32 * k), kIdescN64, (k > K0 || !first) ? 1u : 0u);
}
// D <- A W^T over the input columns [16 K0, 16 K1); a: part 0 in TMEM (parts 32 columns apart), w: part 0 in shared memory.
template <int K0, int K1>
__device__ __forceinline__ void mma_split3(uint32_t one, uint32_t d, uint32_t a, uint32_t w, uint32_t first = 1u) {
  mma_part<K0, K1>(one, d, a + 64, w, first);
  mma_part<K0, K1>(one, d, a + 32, w + kPart, 0u);
  mma_part<K0, K1>(one, d, a, w + 2 * kPart, 0u);
  mma_part<K0, K1>(one, d, a + 32, w, 0u);
  mma_part<K0, K1>(one, d, a, w + kPart, 0u);
  mma_part<K0, K1>(one, d, a, w, 0u);
}
// Layer 2: D <- ones Bias2^T + A W^T (the bias first, like the FP32 sums it replaces)
__device__ __forceinline__ void mma_split3_layer2(uint32_t one, uint32_t d, uint32_t a, uint32_t w, uint32_t ones,
                                                  uint32_t bias) {
  mma_bf16(one, d, sdesc32(ones), sdesc32(bias), kIdescN64, 0u);
  mma_split3<0, 4>(one, d, a, w, 0u);
}
// B's layer 1: the features, and part 0 of the ones columns (its weights are zero on the PE columns)
__device__ __forceinline__ void mma_split3_brdf1(uint32_t one, uint32_t d, uint32_t a, uint32_t w) {
  mma_part<3, 4>(one, d, a, w, 1u);
  mma_split3<0, 2>(one, d, a, w, 0u);
}

__device__ __forceinline__ void tmem_st16x3(uint32_t taddr, const uint32_t (&q0)[16], const uint32_t (&q1)[16],
                                            const uint32_t (&q2)[16]) {
  tmem_st16(taddr, q0);
  tmem_st16(taddr + 32, q1);
  tmem_st16(taddr + 64, q2);
}

// Hidden epilogue: the parts of relu(D[row][0:64]) into the split operand at h_taddr.
__device__ __forceinline__ void epilogue_split3(uint32_t d_taddr, uint32_t h_taddr) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t r[32];
    tmem_ld32(d_taddr + 32 * h, r);
    tmem_ld_wait();
    uint32_t q0[16], q1[16], q2[16];
#pragma unroll
    for (int e = 0; e < 16; ++e)
      split3(fmaxf(__uint_as_float(r[2 * e]), 0.0f), fmaxf(__uint_as_float(r[2 * e + 1]), 0.0f), q0[e], q1[e], q2[e]);
    tmem_st16x3(h_taddr + 16 * h, q0, q1, q2);
  }
}

// The parts of PE(w), with the three ones of the bias in part 0: columns 16..31 of the split layer-1 input.
__device__ __forceinline__ void pe_split3(f3 w, uint32_t (&q0)[16], uint32_t (&q1)[16], uint32_t (&q2)[16]) {
  float pe[32];
  positional_encoding(w, [&](int k, float v) { pe[k] = v; });
#pragma unroll
  for (int k = kPE; k < 32; ++k) pe[k] = (k < kPE + 3) ? 1.0f : 0.0f;
  static_assert(kBiasCol == 32 + kPE, "the ones columns follow the PE");
#pragma unroll
  for (int e = 0; e < 16; ++e) split3(pe[2 * e], pe[2 * e + 1], q0[e], q1[e], q2[e]);
}
__device__ __forceinline__ void store_pe_split3(uint32_t x_taddr, f3 w) {
  uint32_t q0[16], q1[16], q2[16];
  pe_split3(w, q0, q1, q2);
  tmem_st16x3(x_taddr + 16, q0, q1, q2);
}

// I's visibility logit from the FP32 layer-2 accumulator: pairs of hidden units per packed FMA (w in shared memory).
__device__ __forceinline__ float head_vis_s(uint32_t taddr, const float* w, float b) {
  float2 acc = make_float2(b, 0.0f);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t r[32];
    tmem_ld32(taddr + 32 * h, r);
    tmem_ld_wait();
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 ww = *reinterpret_cast<const float4*>(w + 32 * h + 4 * k);
      acc = __ffma2_rn(make_float2(fmaxf(__uint_as_float(r[4 * k]), 0.0f), fmaxf(__uint_as_float(r[4 * k + 1]), 0.0f)),
                       make_float2(ww.x, ww.y), acc);
      acc = __ffma2_rn(make_float2(fmaxf(__uint_as_float(r[4 * k + 2]), 0.0f), fmaxf(__uint_as_float(r[4 * k + 3]), 0.0f)),
                       make_float2(ww.z, ww.w), acc);
    }
  }
  return acc.x + acc.y;
}

}  // namespace rtk
