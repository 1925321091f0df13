// Declarations of the dense-algebra kernels (dense.cu).
#pragma once
#include "internal.h"

namespace sldm {

// One dense system A X = B solved in place (A: n x n, B: n x nrhs, row-major complex64 or complex128).
template <class C>
struct LUSysT {
  C* A;
  C* B;
  int32_t n, nrhs;
};
typedef LUSysT<double2> LUSys;
template <class C>
void lu_solve_batched(const std::vector<LUSysT<C>>& systems, cudaStream_t s);
// Blocked LU of one large system (lu_blocked.cu); lu_solve_batched sends there
// every system of order LU_BLOCKED_MIN or more (below that the look-ahead
// kernel, whose steps need no grid barrier, is faster).
constexpr int LU_BLOCKED_MIN = 1024;
// One or two systems go there from this order on: the look-ahead kernel's chain of
// published columns costs ~18 us a column whatever the order.
constexpr int LU_BLOCKED_FEW = 160;
template <class C>
void lu_solve_blocked(const LUSysT<C>& S, cudaStream_t s);
// C += A B, n x n row-major, the product in FP32
void square_gemm_add(int n, const float2* A, const float2* B, double2* C, cudaStream_t s);
inline void lu_solve_batched(const std::vector<LUSys>& systems, cudaStream_t s) { lu_solve_batched<double2>(systems, s); }

template <class C>
void build_Ml(const sldm_mesh* m, int obj, double k0, const void* LAm, int64_t ldLA, const void* LPm, int64_t ldLP,
              const void* Kl, int64_t ldK, const double* ix_val, C* Ml, C* Rl, cudaStream_t s);

// y = (ar + j ai) A x + beta y over rows [0, m) of a row-major block; x, y hold
// nrhs columns with strides ldx, ldy (entries of the op precision).
struct GemvJob {
  const void* A;
  int64_t lda;
  int32_t m, n;
  const void* x;
  int64_t ldx;
  void* y;
  int64_t ldy;
  double ar, ai;
  int32_t beta, pad;
  // low parts of a complex64 block whose FP64 value is A + Alo (same layout and
  // lda), or null; read only by the FP64-accumulated complex64 product
  const void* Alo;
};
struct TcPlan;
struct X2Plan;
// right-hand sides in lockstep (GMRES) and per pass of the structured product
// and the preconditioner: up to 32 (tensor cores for complex64 operators; the
// CUDA-core kernels take 8 per launch)
constexpr int MAX_NRHS = 32;
constexpr int TILE_NRHS = 8;
struct GemvPlan {
  const char* name = "gemv";   // timer name of its launches
  GemvJob* jobs = nullptr;     // device
  int64_t* rowstart = nullptr; // device, exclusive prefix sum of m
  int njobs = 0;
  int64_t total_rows = 0;
  // tiles of tile_rows rows of one job each (job, first row), device; used
  // with several right-hand sides (null: the one-row-per-warp kernel throughout)
  int2* tiles = nullptr;
  int ntiles = 0;
  int tile_rows = 0;
  // every job carries Alo (complex64 blocks with complex128 vectors only): the
  // product is that of the FP64 operator A + Alo
  bool has_lo = false;
  double bytes = 0;  // matrix bytes one launch streams (its timer's algorithmic units)
  // complex64 blocks and vectors: the tensor-core plan for 9 to 32 right-hand
  // sides per pass (gemm_tc.h), or null / not ok for passes of 8 on the CUDA cores
  const TcPlan* tc = nullptr;
  // FP64-accurate products (has_lo): their tensor-core plan (gemm_x2.h), or null
  const X2Plan* x2 = nullptr;
  // smallest lockstep width sent to the tensor cores (set by gemv_autotune;
  // 33 = never): below it, passes of 8 on the CUDA cores
  int tc_from = TILE_NRHS + 1;
};

// rows per tile of the several-right-hand-side kernel for vectors of es_v bytes
inline int gemv_tile_rows(size_t es_v) { return es_v == 8 ? 32 : 16; }
template <class C>
void gemv_jobs(const GemvPlan& plan, int nrhs, cudaStream_t s);
// complex64 matrix, complex128 vectors, FP64 accumulation
template <class CM, class CV>
void gemv_jobs_mixed(const GemvPlan& plan, int nrhs, cudaStream_t s);
// Measures, on this plan's own blocks, one complex64 pass at 16 and at 32
// right-hand sides on the tensor cores and as passes of 8 on the CUDA cores, and
// sets plan.tc_from to where the tensor cores start to win (9, 17 or 33 =
// never).  The plan's output vectors are overwritten; its inputs must hold
// finite values (the caller zeroes them).
void gemv_autotune(GemvPlan& plan, cudaStream_t s);

// the width forced by sldm_set_tc_policy, 0 = measured
int tc_policy();

struct ApplyDims {
  int32_t ne, nt, nq, nobj;
};
template <class CX, class CY>
struct VecBatch {
  const CX* x[MAX_NRHS] = {};
  CY* y[MAX_NRHS] = {};
  double a[MAX_NRHS] = {};
};
// columns x (blocks scaled by s1, s2, s3) into the structured product's work vectors:
// j, a = j, e, bu = B u, bc = B u (C: the product's precision)
template <class CX, class C>
void apply_in(const sldm_mesh* m, const VecBatch<CX, double2>& x, double s1, double s2, double s3, const ApplyDims& D, void* j,
              void* a, void* e, void* bu, void* bc, int nrhs, cudaStream_t s);
// the product's rows from its work vectors into the columns y (third block scaled by
// s3); with zh, also clears nzh coefficients of every zh[r] and nrm[r]
template <class C, class CY>
void apply_combine(const sldm_mesh* m, const ApplyDims& D, double k0, const double* ix_val, const float2* ix32, const void* z1, const void* z2,
                   const void* w1, const void* w2, const void* w3, const void* e, const void* a, const void* bc, double s3,
                   const VecBatch<double2, CY>& y, int nrhs, cudaStream_t s, double2* const* zh = nullptr, int nzh = 0,
                   double* nrm = nullptr);
// each object's last charge of the columns bc (complex128): minus the sum of its others
void close_charges(const sldm_mesh* m, const ApplyDims& D, void* bc, int nrhs, cudaStream_t s);
// row n of an (n + 1) x nc block = minus the sum of rows 0 .. n - 1
template <class C>
void neg_colsum(C* A, int n, int nc, cudaStream_t s);

// One Gram-Schmidt pass over the Krylov bases of the live right-hand sides of a
// lockstep step: column k of each basis against its columns 0..k-1.  The
// bases have column stride ldv (a multiple of 64) and zero rows n..ldv-1.
struct KrylovStep {
  int64_t n = 0, ldv = 0;
  int k = 0, na = 0;
  void* V[MAX_NRHS] = {};       // basis of right-hand side j (complex64 or complex128)
  double2* h[MAX_NRHS] = {};    // its k projection coefficients (accumulated; cleared by the caller)
  double* nrm = nullptr;        // na squared norms of column k after an update with norm (cleared by the caller)
};
template <class CB>
void krylov_dots(const KrylovStep& ks, cudaStream_t s);                // h_j += V_j[:, :k]^H V_j[:, k]
template <class CB>
void krylov_update(const KrylovStep& ks, bool norm, cudaStream_t s);   // V_j[:, k] -= V_j[:, :k] h_j
template <class C>
void to_c128(const void* src, int64_t n, double2* dst, cudaStream_t s);
// dst = a - b, the difference in FP32
void sub_c64(const float2* a, const float2* b, int64_t n, double2* dst, cudaStream_t s);
// dst = (fl32(src), fl32(src - fl32(src)))
void split_pairs(const double* src, int64_t n, float2* dst, cudaStream_t s);
// hi = complex64 rounding of src, lo = complex64 rounding of src - hi (src = hi + lo to ~2^-48)
void split_c128(const double2* src, int64_t n, float2* hi, float2* lo, cudaStream_t s);
// dst += lo (complex64 low parts onto a complex128 copy of the high parts)
void add_lo_c128(const float2* lo, int64_t n, double2* dst, cudaStream_t s);
template <class C>
void copy_scaled(const void* src, int64_t n, double alpha, void* dst, cudaStream_t s);
// Copies of sub-blocks within one row-major matrix (leading dimension ld):
// rows [sr, sr + nr) x cols [sc, sc + nc) to [dr, dr + nr) x [dc, dc + nc).
// With `transpose` the source's transpose goes to rows [dr, dr + nc) x cols [dc, dc + nr).
// Sources are never destinations of the same call.
struct BlockCopy {
  int32_t sr, sc, dr, dc, nr, nc;
};
void copy_blocks(const std::vector<BlockCopy>& copies, size_t esz, void* M, int64_t ld, cudaStream_t s,
                 bool transpose = false);
template <class C>
void add_ix(const sldm_mesh* m, int obj, double alpha, const double* ix_val, void* K, int64_t ld, cudaStream_t s);

// ---------------------------------------------------------------- GMRES on the device
// Per right-hand side r of a lockstep GMRES cycle: iterations, columns in use,
// whether it still iterates, ||b|| and the cycle's starting residual.
struct GmresState {
  int32_t it, kused, live, pad;
  double bnorm, beta;
};
// Step k of the Arnoldi process for the na active right-hand sides on[j]:
// column k of H_r from the two Gram-Schmidt passes (dh + r * ldh: coefficients
// of pass one at [0, k], pass two at [m + 2, m + 2 + k]) and h_{k+1,k} =
// sqrt(nrm[j]); the earlier Givens rotations, a new one annihilating h_{k+1,k},
// the rotated residual vector g_r; then the convergence tests (|g_{k+1}| <=
// tol ||b||, it >= maxit, h_{k+1,k} = 0, and with refine |g_{k+1}| <= cycle
// beta) clear live.  flags[r] (pinned host memory) receives whether r still iterates.
// H: (m + 1) x m row-major per right-hand side, cs, sn: m, g: m + 1 (complex).
struct GivensArgs {
  int k, m, na, refine;
  int on[MAX_NRHS];
  const double2* dh;
  int64_t ldh;
  const double* nrm;
  double2 *H, *cs, *sn, *g;
  GmresState* st;
  double tol, cycle;
  int maxit, pad;
  int32_t* flags;
};
// w_j (column ks.k of its basis) orthogonalised twice against columns 0 .. ks.k - 1, column
// ks.k - 1 = a.k of H, the rotations and tests, and w_j / h_{k+1,k}: one launch of a cluster per
// right-hand side for small systems, else separate kernels, which add up in h1[j] and
// h2[j] (a.dh's two parts) and a.nrm (cleared by the caller).
template <class CB>
void gmres_orthogonalise(const GivensArgs& a, KrylovStep ks, double2* const* h1, double2* const* h2, cudaStream_t s);
// b = D b, r = b, nrm[c] += |b_c|^2 (D = diag(1, l) with l from entry n2 on; nr columns of n)
void gmres_rhs(int64_t n, int64_t n2, double l, double2* b, double2* r, double* nrm, int nr, cudaStream_t s);
// r = b - y, nrm[c] += |r_c|^2
void gmres_residual(int64_t n, const double2* b, const double2* y, double2* r, double* nrm, int nr, cudaStream_t s);
// A cycle's state and g of every column; v0 = r / beta of the live ones
struct CycleStart {
  int it[MAX_NRHS], live[MAX_NRHS];
  double bnorm[MAX_NRHS], beta[MAX_NRHS];
  void* v0[MAX_NRHS];
  const double2* r;
  GmresState* st;
  double2* g;
  int m;
};
template <class CB>
void gmres_cycle_start(int64_t n, const CycleStart& a, int nr, cudaStream_t s);
// y_r = H_r^-1 g_r (upper triangular, k[j] columns) into dh + r * ldh and out[j] = V[j] y_r for
// the na right-hand sides r = on[j]
struct CycleEnd {
  int on[MAX_NRHS], k[MAX_NRHS];
  void* V[MAX_NRHS];
  double2* out[MAX_NRHS];
  const double2 *H, *g;
  double2* dh;
  int64_t ldh, ldv;
  int m;
};
template <class CB>
void gmres_cycle_end(int64_t n, const CycleEnd& a, int na, cudaStream_t s);
// y_j += diag(s1, 1, s3) x_j
void gmres_add_scaled(int64_t n, int64_t ne, double s1, double s3, const VecBatch<double2, double2>& b, int na, cudaStream_t s);

}  // namespace sldm
