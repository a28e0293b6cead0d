// The two fp16 planes of a value: what the tensor-core products read (gemm_tc.cuh says why two).
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace pd {

__device__ __forceinline__ float tc_pow2(int e) { return __uint_as_float((uint32_t)(e + 127) << 23); }

// One scaled value -> its two planes (as floats that fp16 holds exactly inside the normal range).
__device__ __forceinline__ void tc_split(float x, float scale, float &hi, float &lo) {
  const float xs = x * scale;
  hi = __uint_as_float((__float_as_uint(xs) + 0x1000u) & 0xFFFFE000u);     // 11 significant bits, nearest
  lo = (xs - hi) * 2048.0f;
}
__device__ __forceinline__ uint32_t tc_pack(float a, float b) {
  const __half2 v = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}
// Four / eight consecutive values -> 8 / 16 bytes of the hi plane and of the lo plane.
__device__ __forceinline__ void tc_split4(float4 x, float scale, uint2 &h, uint2 &l) {
  float hi[4], lo[4];
  tc_split(x.x, scale, hi[0], lo[0]); tc_split(x.y, scale, hi[1], lo[1]);
  tc_split(x.z, scale, hi[2], lo[2]); tc_split(x.w, scale, hi[3], lo[3]);
  h = make_uint2(tc_pack(hi[0], hi[1]), tc_pack(hi[2], hi[3]));
  l = make_uint2(tc_pack(lo[0], lo[1]), tc_pack(lo[2], lo[3]));
}
__device__ __forceinline__ void tc_split8(float4 a, float4 b, float scale, uint4 &h, uint4 &l) {
  uint2 h0, l0, h1, l1;
  tc_split4(a, scale, h0, l0);
  tc_split4(b, scale, h1, l1);
  h = make_uint4(h0.x, h0.y, h1.x, h1.y);
  l = make_uint4(l0.x, l0.y, l1.x, l1.y);
}
// An exponent outside the normal range (TC_NO_PREDICTION) scales by 1: planes made with it are refused by the product.
__device__ __forceinline__ float tc_scale_of(int e) { return tc_pow2(e < -100 || e > 100 ? 0 : e); }


}  // namespace pd
