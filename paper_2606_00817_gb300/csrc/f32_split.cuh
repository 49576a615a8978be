// f32_split.cuh -- an FP32 value as three bf16 values that add up to it, for
// FP32 products on the bf16 tensor cores (tc_gemm_f32.cu).
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

namespace ddf {

// x = x0 + x1 + x2: x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1),
// rounded to nearest; both differences are exact in FP32, and so is x2, unless
// it falls below bf16's subnormals (an error under 2^-133). Beyond bf16's
// largest value x0 is that value instead of infinity. An infinity or a NaN is
// carried by x2 alone, the piece that is multiplied by the other operand's first
// piece only: beside x0 it would meet second and third pieces of either sign or
// zero, and an infinite activation would come out as NaN instead of infinity
// times its weight.
__device__ __forceinline__ void f32_split(float x, float& x0, float& x1, float& x2) {
  x0 = __bfloat162float(__float2bfloat16_rn(x));
  if (fabsf(x0) == __int_as_float(0x7f800000)) x0 = __int_as_float(__float_as_int(x) & 0xffff0000);
  const float r1 = x - x0;
  x1 = __bfloat162float(__float2bfloat16_rn(r1));
  x2 = r1 - x1;
  if (!(fabsf(x) < __int_as_float(0x7f800000))) {
    x0 = x1 = 0.f;
    x2 = x;
  }
}

// The three pieces of 8 consecutive values, packed as 8 bf16 each.
__device__ __forceinline__ void f32_split8(const float* x, uint4 (&w)[3]) {
  uint32_t r[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float a[3], b[3];
    f32_split(x[2 * i], a[0], a[1], a[2]);
    f32_split(x[2 * i + 1], b[0], b[1], b[2]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const __nv_bfloat162 v = __floats2bfloat162_rn(a[j], b[j]);
      r[j][i] = *reinterpret_cast<const uint32_t*>(&v);
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) w[j] = make_uint4(r[j][0], r[j][1], r[j][2], r[j][3]);
}

}  // namespace ddf
