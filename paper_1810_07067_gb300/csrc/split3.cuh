// An FP32 value as the exact sum of three BF16 pieces (24 bits).
#pragma once
#include <cuda_bf16.h>

__device__ __forceinline__ void split3(float x, __nv_bfloat16* p) {
  __nv_bfloat16 h = __float2bfloat16_rn(x);
  float r1 = x - __bfloat162float(h);
  __nv_bfloat16 m = __float2bfloat16_rn(r1);
  float r2 = r1 - __bfloat162float(m);
  p[0] = h; p[1] = m; p[2] = __float2bfloat16_rn(r2);
}
