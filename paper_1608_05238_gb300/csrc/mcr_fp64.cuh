// mcr_fp64.cuh -- FP64 helpers of the per-pixel and per-voxel sums.
#pragma once

namespace mcr {

// A normal float as a double by integer operations (the conversion itself takes a slot of the FP64 pipe,
// which does 1/64 of the FP32 rate on this part); `special` is set for zeros, subnormals, infinities and NaN.
__device__ __forceinline__ double widen_normal(float x, bool &special) {
  const unsigned u = __float_as_uint(x);
  special |= ((u + 0x00800000u) & 0x7F000000u) == 0u;  // exponent 0 or 255
  return __hiloint2double((int)((((int)u >> 3) & 0x8FFFFFFF) + 0x38000000), (int)(u << 29));
}

}  // namespace mcr
