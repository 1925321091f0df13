// Exact float -> double without the FP64 pipe.
#pragma once
#include <cuda_runtime.h>

namespace sldm {

// Float to double on the integer pipe: the conversion instruction issues on this
// part's FP64 pipe (two per SM and clock), which these kernels keep for their FMAs.
// Exact; denormals become zero.
__device__ __forceinline__ double widen(float v) {
  const unsigned b = __float_as_uint(v), e = b & 0x7f800000u;
  unsigned hi = ((b & 0x7fffffffu) >> 3) + 0x38000000u;
  if (e == 0) hi = 0;
  if (e == 0x7f800000u) hi |= 0x7ff00000u;
  return __hiloint2double(int(hi | (b & 0x80000000u)), e == 0 ? 0 : int(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

}  // namespace sldm
