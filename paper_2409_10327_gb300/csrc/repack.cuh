// The device images of both MLPs' weights, element by element from the
// caller's canonical blobs: the FP32 image (rt_internal.h's OFF_*) and the
// BF16 image (OFFB_*).
#pragma once

#include <cuda_bf16.h>

#include "rt_internal.h"

namespace rtk {

// Canonical blob (per MLP): W1 [64][in], b1 [64], W2 [64][64], b2 [64],
// W3 [out][64], b3 [out].  Element e of the transposed FP32 image.
__device__ __forceinline__ float packed_value(const float* __restrict__ bw, const float* __restrict__ iw, int lf, int e) {
  const int in_i = lf + kPE;
  // I blob offsets
  const int iW1 = 0, iB1 = iW1 + 64 * in_i, iW2 = iB1 + 64, iB2 = iW2 + 64 * 64, iW3 = iB2 + 64, iB3 = iW3 + 2 * 64;
  // B blob offsets
  const int bW1 = 0, bB1 = bW1 + 64 * lf, bW2 = bB1 + 64, bB2 = bW2 + 64 * 64, bW3 = bB2 + 64, bB3 = bW3 + 7 * 64;
  float v = 0.0f;
  if (e < OFF_IW1P) {                         // I W1, feature rows [k][c]
    const int k = (e - OFF_IW1F) / 64, c = (e - OFF_IW1F) % 64;
    if (k < lf) v = iw[iW1 + c * in_i + k];
  } else if (e < OFF_IB1) {                   // I W1, PE rows
    const int k = (e - OFF_IW1P) / 64, c = (e - OFF_IW1P) % 64;
    if (k < kPE) v = iw[iW1 + c * in_i + lf + k];
  } else if (e < OFF_IW2) {
    v = iw[iB1 + (e - OFF_IB1)];
  } else if (e < OFF_IB2) {
    const int k = (e - OFF_IW2) / 64, c = (e - OFF_IW2) % 64;
    v = iw[iW2 + c * 64 + k];
  } else if (e < OFF_IW3) {
    v = iw[iB2 + (e - OFF_IB2)];
  } else if (e < OFF_IB3) {
    const int k = (e - OFF_IW3) / 2, c = (e - OFF_IW3) % 2;
    v = iw[iW3 + c * 64 + k];
  } else if (e < OFF_BW1) {
    const int c = e - OFF_IB3;
    if (c < 2) v = iw[iB3 + c];
  } else if (e < OFF_BB1) {
    const int k = (e - OFF_BW1) / 64, c = (e - OFF_BW1) % 64;
    if (k < lf) v = bw[bW1 + c * lf + k];
  } else if (e < OFF_BW2) {
    v = bw[bB1 + (e - OFF_BB1)];
  } else if (e < OFF_BB2) {
    const int k = (e - OFF_BW2) / 64, c = (e - OFF_BW2) % 64;
    v = bw[bW2 + c * 64 + k];
  } else if (e < OFF_BW3) {
    v = bw[bB2 + (e - OFF_BB2)];
  } else if (e < OFF_BB3) {
    const int k = (e - OFF_BW3) / 8, c = (e - OFF_BW3) % 8;
    if (c < 7) v = bw[bW3 + c * 64 + k];
  } else {
    const int c = e - OFF_BB3;
    if (c < 7) v = bw[bB3 + c];
  }
  return v;
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(v);
  lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// The bf16 at byte offset `byte` of the BF16 image; wp(e) is element e of the FP32 image.
template <class W>
__device__ __forceinline__ __nv_bfloat16 bf16_image_value(int byte, W wp) {
  __nv_bfloat16 v = __float2bfloat16_rn(0.0f);
  if (byte < OFFB_IB2 || byte >= OFFB_IW1L) {
    // one of the six 64 x 64 swizzled matrices: invert swz128
    const int tile = byte < OFFB_IB2 ? byte / 8192 : 4 + (byte - OFFB_IW1L) / 8192;
    const int o = byte % 8192;
    const int n = (o / 1024) * 8 + (o % 1024) / 128;
    const int chunk = ((o % 128) / 16) ^ (n & 7);
    const int k = chunk * 8 + (o % 16) / 2;
    float f = 0.0f;
    if (tile == 0 || tile == 4) {                       // I layer 1: [f | PE | 1 | 1 | 0]
      f = k < 32 ? wp(OFF_IW1F + k * 64 + n) : (k < kBiasCol ? wp(OFF_IW1P + (k - 32) * 64 + n) : 0.0f);
    } else if (tile == 1 || tile == 5) {
      f = wp(OFF_IW2 + k * 64 + n);
    } else if (tile == 2) {                             // B layer 1: [f | 0 | b1]
      if (k < 32) f = wp(OFF_BW1 + k * 64 + n);
    } else {
      f = wp(OFF_BW2 + k * 64 + n);
    }
    v = __float2bfloat16_rn(f);
    if (tile >= 4) {                                    // the rounding residual of the hi tile
      __nv_bfloat16 hi, lo;
      split_bf16(f, hi, lo);
      v = lo;
    }
    if (tile == 0 || tile == 2) {
      const float b = tile == 0 ? wp(OFF_IB1 + n) : wp(OFF_BB1 + n);
      __nv_bfloat16 hi, lo;
      split_bf16(b, hi, lo);
      if (k == kBiasCol) v = hi;
      if (k == kBiasCol + 1) v = lo;
    }
  } else if (byte < OFFB_ONES) {
    // layer-2 bias tiles: row n = 8 x hi/8, 8 x lo/8 (exact scalings by 1/8)
    const int tile = (byte - OFFB_IB2) / 2048, o = (byte - OFFB_IB2) % 2048;
    const int n = o / 32, k = (o % 32) / 2;
    const float b = tile == 0 ? wp(OFF_IB2 + n) : wp(OFF_BB2 + n);
    __nv_bfloat16 hi, lo;
    split_bf16(b, hi, lo);
    v = __float2bfloat16_rn(0.125f * __bfloat162float(k < 8 ? hi : lo));
  } else {
    v = __float2bfloat16_rn(1.0f);                      // the all-ones tile
  }
  return v;
}

}  // namespace rtk
