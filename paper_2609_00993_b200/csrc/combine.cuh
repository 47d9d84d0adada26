// The arithmetic of the combine (a9): a token's sum in fp32, eight columns at a time, rounded once to bf16.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace moe {

// acc += w * v for eight bf16 values; a bf16 widens to fp32 by a 16-bit shift (low half) or a mask (high half)
__device__ __forceinline__ void fma_bf16x8(float (&acc)[8], const uint4& v, float w) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    acc[2 * q] = fmaf(w, __uint_as_float(u[q] << 16), acc[2 * q]);
    acc[2 * q + 1] = fmaf(w, __uint_as_float(u[q] & 0xffff0000u), acc[2 * q + 1]);
  }
}

__device__ __forceinline__ uint4 bf16x8(const float (&acc)[8]) {
  uint4 o;
  __nv_bfloat162* oh = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
  for (int q = 0; q < 4; ++q) oh[q] = __floats2bfloat162_rn(acc[2 * q], acc[2 * q + 1]);
  return o;
}

}  // namespace moe
