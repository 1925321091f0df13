// Preconditioner P of Eq. pcext (precond.cu).
#pragma once
#include "dense.h"
#include "gemm_tc.h"

namespace sldm {

// Object description for the preconditioner (offsets are elements of the op's local block storage).
struct PrecObj {
  int32_t e0, ne, t0, nt, q0;
  int32_t same;  // the first object with the same Schur complement (a repeat of this one's blocks), or itself
  int64_t oLA, oK, oLP;
};

struct Precond {
  DBuf<PrecObj> objs;
  DBuf<double2> lam;    // 4 per edge: Lambda11, Lambda12, Lambda21, Lambda22
  DBuf<float4> lam32, pdiag32;  // complex64 operators: both as pairs (hi.x, hi.y, lo.x, lo.y)
  DBuf<double2> pdiag;  // 2 per triangle: diag L^phi_m, diag of the object's L^phi/eps
  // per object nt_o x (nt_o - 1): B_o S_o^-1 = [S_o^-1; minus its column sums], row-major, so
  // that the product gives the full charges B x3 (complex128 operators)
  DBuf<double2> sinv;
  DBuf<float2> sinv32;  // the same in complex64 (complex64 operators: an FP32 preconditioner)
  bool f32 = false;
  // WR columns each, entries of the preconditioner's precision: t3 of nq, bx = B x3 of nt
  DBuf<double2> t3, bx;
  int64_t nq = 0;
  DBuf<GemvJob> jobs;
  DBuf<int64_t> rs;
  DBuf<int2> tiles;
  GemvPlan plan;
  TcPlan tc;  // complex64: the Schur-inverse products on the tensor cores (9 to 32 columns)
  bool ready = false;
  size_t bytes() const { return bytes_of(objs, lam, lam32, pdiag32, pdiag, sinv, sinv32, t3, bx, jobs, rs, tiles, tc); }
};

template <class C>
void prec_setup(Precond& P, const sldm_mesh* m, const std::vector<PrecObj>& objs, double k0, const void* LAm,
                const void* LPm, const char* loc, const double* ix_val, cudaStream_t s);
// Columns of x = P^-1 D r, D = diag(1, 1, s3), for nr <= MAX_NRHS columns r.x (CX), either
// into the work vectors of the structured product (C: its precision; j, a = j, e, bu =
// B u, bc = B u) or added to the columns r.y (complex128).
template <class CX, class C>
void prec_apply_in(const Precond& P, const sldm_mesh* m, const VecBatch<CX, double2>& r, double s3, void* j, void* a, void* e,
                   void* bu, void* bc, int nr, cudaStream_t s);
void prec_apply_add(const Precond& P, const sldm_mesh* m, const VecBatch<double2, double2>& r, double s3, int nr,
                    cudaStream_t s);

}  // namespace sldm
