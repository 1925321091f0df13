// Exact float -> double without the FP64 pipe.
#pragma once
#include <cuda_runtime.h>

namespace sldm {

// Float to double on the integer pipe: the conversion instruction issues on this
// part's FP64 pipe (two per SM and clock), which these kernels keep for their FMAs.
// Exact for every class of number: denormals are brought into the normal range by 2^64 first (exact in
// FP32) and their exponent taken back in the bias.
__device__ __forceinline__ double widen(float v) {
  unsigned b = __float_as_uint(v), bias = 0x38000000u;
  if ((b & 0x7f800000u) == 0) {  // zero or denormal
    b = __float_as_uint(__fmul_rn(v, 0x1p64f));
    bias = (b << 1) == 0 ? 0u : 0x34000000u;
  }
  unsigned hi = ((b & 0x7fffffffu) >> 3) + bias;
  if ((b & 0x7f800000u) == 0x7f800000u) hi |= 0x7ff00000u;
  return __hiloint2double(int(hi | (b & 0x80000000u)), int(b << 29));
}
__device__ __forceinline__ double widen(double v) { return v; }

}  // namespace sldm
