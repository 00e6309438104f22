// Integer slices of FP32 values for the tensor cores (gemm_f32tc.cu): shared by
// the kernels that write the operands.
#pragma once

#include "kernels.cuh"

namespace gcnn {
namespace {
// ---------------------------------------------------------------- slices
// Scale of a row or column with largest magnitude m < 2^e: inv = 2^(8-e) brings
// it to at most 256; the result's factor is 2^(e-8).  Entries below 2^-118 keep
// the scale of 2^-118; a NaN or an infinity gives a NaN factor.
__device__ __forceinline__ void slice_scale(float m, float *inv, float *factor) {
  const unsigned b = __float_as_uint(m);
  if ((b & 0x7f800000u) == 0x7f800000u) {
    *inv = 0.f;
    *factor = __uint_as_float(0x7fc00000u);
    return;
  }
  const int e = max((int)(b >> 23) - 126, -118);
  *inv = __uint_as_float((unsigned)(135 - e) << 23);
  *factor = __uint_as_float((unsigned)(119 + e) << 23);
}

// v = inv x as s1 + s2 2^-9 + s3 2^-18 (every step exact but the last rounding)
__device__ __forceinline__ void slice3(float v, float s[3]) {
  s[0] = rintf(v);
  const float r = (v - s[0]) * 512.f;
  s[1] = rintf(r);
  s[2] = rintf((r - s[1]) * 512.f);
}

__device__ __forceinline__ float max4(float m, float4 v) {
  // a NaN must win: fmaxf would drop it
  const float a = fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w)));
  const bool nan = v.x != v.x || v.y != v.y || v.z != v.z || v.w != v.w;
  return nan ? __uint_as_float(0x7f800000u) : fmaxf(m, a);
}

// The three slices of four entries at o, o + width and o + 2 width (BF16, exact).
__device__ __forceinline__ void store_slices(float4 v, float inv, uint16_t *o, int width) {
  float a[3], b[3], c[3], e[3];
  slice3(v.x * inv, a);
  slice3(v.y * inv, b);
  slice3(v.z * inv, c);
  slice3(v.w * inv, e);
#pragma unroll
  for (int p = 0; p < 3; ++p) st_bf16x4(o + (size_t)p * width, a[p], b[p], c[p], e[p]);
}

}  // namespace
}  // namespace gcnn
