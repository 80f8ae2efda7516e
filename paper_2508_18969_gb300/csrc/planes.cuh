// FP32 values as three BF16 planes (mlp_split.cu).
#pragma once

#include <cuda_bf16.h>

namespace dfgb {

// The three BF16 planes of one FP32 value. Infinities and NaN stay in plane 0; a finite value that
// would round to a BF16 infinity is truncated there instead (the remainder stays exact).
__device__ __forceinline__ void split_one(float v, __nv_bfloat16& h0, __nv_bfloat16& h1,
                                          __nv_bfloat16& h2) {
  h0 = __float2bfloat16_rn(v);
  float r = v - __bfloat162float(h0);
  if (!(fabsf(r) <= 3.0e38f)) {
    if (!isfinite(v)) {
      h1 = h2 = __float2bfloat16_rn(0.0f);
      return;
    }
    h0 = __ushort_as_bfloat16((unsigned short)(__float_as_uint(v) >> 16));
    r = v - __bfloat162float(h0);
  }
  h1 = __float2bfloat16_rn(r);
  h2 = __float2bfloat16_rn(r - __bfloat162float(h1));
}

}  // namespace dfgb
