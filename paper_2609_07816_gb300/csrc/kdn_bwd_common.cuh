// kdn_bwd_common.cuh -- operand-tile and gradient-store helpers shared by the fused
// backward sweeps (kdn_fused_bwd.cu, kdn_split_bwd.cu).
#pragma once

#include "kdn_fused_common.cuh"

namespace kdn {
namespace fused {

__device__ __forceinline__ uint64_t kdesc(const unsigned char *p) {
  return sw128_desc(smem_u32(p), 16, 1024);
}
__device__ __forceinline__ uint64_t mdesc(const unsigned char *p, uint32_t lbo) {
  return sw128_desc(smem_u32(p), lbo, 1024);
}
// x ~ hi + lo, both fp16: returns hi, writes the lo chunk
__device__ __forceinline__ uint4 split_h8(const float *x, uint4 *lo) {
  float h[8], l[8];
  const uint4 hi = pack_h8(x);
  unpack_h8(hi, h);
#pragma unroll
  for (int j = 0; j < 8; ++j) l[j] = x[j] - h[j];
  *lo = pack_h8(l);
  return hi;
}

// Row `row` of a [128][64] 16-bit tile (one 128-byte-swizzled slab), tokens
// 16 q .. 16 q + 15: two 16-byte chunks.
__device__ __forceinline__ void st_row16_bf(unsigned char *tile, int row, int q, const float *v) {
  sm16(tile, chunk_off(row, 2 * q)) = pack_bf8(v);
  sm16(tile, chunk_off(row, 2 * q + 1)) = pack_bf8(v + 8);
}
__device__ __forceinline__ void st_row16_h(unsigned char *tile, int row, int q, const float *v) {
  sm16(tile, chunk_off(row, 2 * q)) = pack_h8(v);
  sm16(tile, chunk_off(row, 2 * q + 1)) = pack_h8(v + 8);
}
__device__ __forceinline__ void st_row16_split(unsigned char *hi, unsigned char *lo, int row, int q,
                                               const float *v) {
  uint4 l0, l1;
  sm16(hi, chunk_off(row, 2 * q)) = split_bf8(v, &l0);
  sm16(hi, chunk_off(row, 2 * q + 1)) = split_bf8(v + 8, &l1);
  sm16(lo, chunk_off(row, 2 * q)) = l0;
  sm16(lo, chunk_off(row, 2 * q + 1)) = l1;
}

// Reduce-scatter of 16 per-lane values over a warp: returns, in lanes 2j and
// 2j + 1, the warp-wide sum of v[j].
__device__ __forceinline__ float rs16(const float *v, int lane) {
  float w8[8], w4[4], w2[2];
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float keep = b4 ? v[8 + j] : v[j], send = b4 ? v[j] : v[8 + j];
    w8[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float keep = b3 ? w8[4 + j] : w8[j], send = b3 ? w8[j] : w8[4 + j];
    w4[j] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const float keep = b2 ? w4[2 + j] : w4[j], send = b2 ? w4[j] : w4[2 + j];
    w2[j] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
  }
  const float keep = b1 ? w2[1] : w2[0], send = b1 ? w2[0] : w2[1];
  const float w1 = keep + __shfl_xor_sync(0xffffffffu, send, 2);
  return w1 + __shfl_xor_sync(0xffffffffu, w1, 1);
}

// Output store in the gradient dtype (OBF: bfloat16, else float32).  float32
// gradients are written with the streaming hint: they are not read again by this
// kernel, and evicting them first keeps L2 for the context records it prefetches.
template <int OBF>
__device__ __forceinline__ void st_grad(void *p, size_t i, float x) {
  if (OBF) static_cast<__nv_bfloat16 *>(p)[i] = __float2bfloat16_rn(x);
  else __stcs(static_cast<float *>(p) + i, x);
}

}  // namespace fused
}  // namespace kdn
