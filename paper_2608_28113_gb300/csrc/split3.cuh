// split3.cuh -- fp32 values as three bf16 parts for the split-operand GEMMs (update.cu).
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

namespace hscale {

// x = x1 + x2 + x3 with bf16 parts, each difference exact in fp32: the parts carry x to
// about 2^-24 relative.
__device__ __forceinline__ void split3(float x, uint16_t (&p)[3]) {
  const __nv_bfloat16 a = __float2bfloat16_rn(x);
  const float r1 = __fsub_rn(x, __bfloat162float(a));
  const __nv_bfloat16 b = __float2bfloat16_rn(r1);
  const float r2 = __fsub_rn(r1, __bfloat162float(b));
  const __nv_bfloat16 c = __float2bfloat16_rn(r2);
  p[0] = __bfloat16_as_ushort(a);
  p[1] = __bfloat16_as_ushort(b);
  p[2] = __bfloat16_as_ushort(c);
}

// The parts of four consecutive values: 8 bytes in each of the three segments, seg elements
// apart, at dst (8-byte aligned).
__device__ __forceinline__ void store_split3x4(uint16_t* dst, int64_t seg, const float (&v)[4]) {
  uint16_t p[4][3];
#pragma unroll
  for (int t = 0; t < 4; ++t) split3(v[t], p[t]);
#pragma unroll
  for (int s = 0; s < 3; ++s)
    *reinterpret_cast<uint2*>(dst + s * seg) = make_uint2((uint32_t)p[0][s] | ((uint32_t)p[1][s] << 16),
                                                          (uint32_t)p[2][s] | ((uint32_t)p[3][s] << 16));
}

}  // namespace hscale
