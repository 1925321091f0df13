// Sums of products in pairs of FP32 numbers: ~48 bits without the FP64 pipe, whose instructions cost 64
// FP32 ones on this part.  For the sparse parts of complex64 products, whose terms are FP32
// numbers times FP64 coefficients held as hi + lo (split_pairs).  Below 2^-101 a product's own
// rounding error falls under FP32's smallest number: an error of 2^-149 per operation then, the spacing of
// the terms themselves.  A sum that overflows or holds an infinity is that infinity (its error
// would be Inf - Inf), a NaN stays NaN.
#pragma once
#include <cuda_runtime.h>

#include "widen.cuh"

namespace sldm {

struct P32 {
  float s = 0.f, c = 0.f;  // the sum and its error
  __device__ __forceinline__ void add(float v) {  // TwoSum
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
  }
  // += (h + l) v
  __device__ __forceinline__ void fma(float h, float l, float v) {
    const float p = __fmul_rn(h, v);
    c = __fadd_rn(c, __fmaf_rn(l, v, __fmaf_rn(h, v, -p)));
    add(p);
  }
  // += (h + l) v
  __device__ __forceinline__ void fma(float h, float l, const P32& v) {
    const float p = __fmul_rn(h, v.s);
    c = __fadd_rn(c, __fmaf_rn(h, v.c, __fmaf_rn(l, v.s, __fmaf_rn(h, v.s, -p))));
    add(p);
  }
  __device__ __forceinline__ P32 scaled(float h, float l) const {
    P32 r;
    r.fma(h, l, *this);
    return r;
  }
  __device__ __forceinline__ float err() const { return fabsf(s) < __int_as_float(0x7f800000) ? c : 0.f; }
  __device__ __forceinline__ void get(float& o) const { o = __fadd_rn(s, err()); }
  __device__ __forceinline__ void get(double& o) const { o = widen(s) + widen(err()); }
};
// complex += a v, a = (hi.x + lo.x) + j (hi.y + lo.y) as (hi.x, hi.y, lo.x, lo.y)
template <class V>
__device__ __forceinline__ void cfma_pair(P32& re, P32& im, const float4 a, const V& vx, const V& vy) {
  re.fma(a.x, a.z, vx);
  re.fma(-a.y, -a.w, vy);
  im.fma(a.x, a.z, vy);
  im.fma(a.y, a.w, vx);
}

}  // namespace sldm
