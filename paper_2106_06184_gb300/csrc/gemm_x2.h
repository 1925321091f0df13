// FP64-accurate multi-right-hand-side products of complex64 block pairs on the tensor
// cores (gemm_x2.cu).
#pragma once
#include "gemm_tc.h"

namespace sldm {

constexpr int X2_NRHS = 16;  // right-hand sides of one pass

// Beside the complex64 plan of the same jobs (same blocks, same order), whose tiles,
// CTA assignment and scale exponents it uses: the tensor maps of the low parts and the
// digits of the right-hand sides, rebuilt for each pass.
struct X2Plan {
  const TcPlan* tc = nullptr;
  DBuf<unsigned char> lomaps, bmap;
  DBuf<uint16_t> bprime;
  DBuf<float> bscale;
  int from = X2_NRHS + 1;  // right-hand sides a pass is worth it for
  bool ok = false;
  size_t bytes() const { return bytes_of(lomaps, bmap, bprime, bscale); }
};
void x2_plan_build(const std::vector<GemvJob>& jobs, const TcPlan& tc, X2Plan& xp, cudaStream_t s);
// Y = alpha (A + Alo) X (+ Y) for nrhs <= 16 complex128 columns from col0
void gemm_x2(const GemvPlan& plan, const X2Plan& xp, int nrhs, int col0, cudaStream_t s);

}  // namespace sldm
