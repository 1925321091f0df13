// Multi-right-hand-side complex64 block products on the 5th-generation tensor
// cores (gemm_tc.cu): Y = alpha A X (+ Y) for 9 to 32 right-hand sides per pass.
#pragma once
#include "dense.h"

namespace sldm {

// Right-hand sides one tensor-core pass takes (accumulator width 2 x 32 FP32 columns).
constexpr int TC_MAX_NRHS = 32;

// 128 rows of a job from row0, over K sub-chunks [k0, k0 + nk) of 32 FP32
// columns (whole stages); split: one of two K halves of the rows, added into Y
struct TcTile {
  int32_t job, row0, k0, nk, split;
};

// A job's scale exponents (offset, rows padded to whole tiles) and its first B' box
struct TcJob {
  int64_t aexp;
  int32_t mpad, base;
};

// Per GEMV plan: one TMA tensor map per job (the block seen as a row-major FP32
// matrix of m rows and 2n columns), the 128-row tiles of every job (long ones in
// two K halves), and their assignment to CTAs (longest first, to the least loaded CTA); the real-form
// right-hand-side operand B' of every stage, rebuilt for each pass.
struct TcPlan {
  DBuf<unsigned char> maps;  // 128-byte tensor maps, 64-byte aligned
  DBuf<TcTile> tiles;
  DBuf<int32_t> cta_begin;   // CTA c takes tiles [cta_begin[c], cta_begin[c + 1])
  DBuf<int> err;             // set to 1 by a CTA whose bounded wait ran out
  mutable bool ran = false;  // passes launched since err was last read
  // B' of the pass (built from the vectors before each pass): stage g of the plan is
  // (job gjob[g], its stage gst[g]); boxes of 128 rows (hi, lo) x 128 bytes, two per stage in FP16,
  // four in TF32, read by TMA through bmap, and (FP16) the factor that undoes each right-hand side's scale
  bool f16 = true;           // operands as scaled FP16 pairs, or TF32 pairs
  DBuf<unsigned char> bprime;
  DBuf<float> bscale;
  DBuf<unsigned char> bmap;
  DBuf<int32_t> gjob, gst;
  // scale exponents of A by job, stage and row (set when the plan is built)
  DBuf<TcJob> tj;
  DBuf<signed char> aexp;
  DBuf<TcTile> ztiles;       // the first halves of the split tiles (their Y rows are zeroed per pass)
  int nstage = 0, nzero = 0;
  int nctas = 0;
  int longest = 0;           // stages of the CTA with the most
  bool ok = false;           // every job fits the tensor-core path
  size_t bytes() const { return bytes_of(maps, tiles, cta_begin, err, bprime, bscale, bmap, gjob, gst, tj, aexp, ztiles); }
};

// Builds tp for the jobs of a complex64 plan (host copies of the jobs), whose blocks
// are filled already (their scale exponents are read off).  tp.ok is
// false (and the plan keeps the CUDA-core kernels) when a job's row pitch is
// not a multiple of 16 bytes or the driver's tensor-map encoder is unavailable.
//
// f16: the FP16 form; else TF32, no more accurate and slower (8 x 8 metasurface, 32 right-hand
// sides: 1,390 against 1,610 us), for products whose rounding shows in complex128 results.
void tc_plan_build(const std::vector<GemvJob>& jobs, TcPlan& tp, bool f16, cudaStream_t s);
// 128-byte TMA map of a 2-D array (CUtensorMapDataType type, nx x ny, row pitch in bytes,
// boxes bx x by, 128-byte swizzle), and of a complex64 block read as FP32 in boxes of
// 32 columns x 128 rows; false where the array cannot be mapped
bool tc_map_2d(int type, const void* p, uint64_t nx, uint64_t ny, uint64_t pitch, int bx, int by, unsigned char* out);
bool tc_block_map(const void* A, int64_t lda, int m, int n, unsigned char* out);
// One pass over every job of `plan` for nrhs (<= 32) right-hand sides.
void gemm_tc(const GemvPlan& plan, const TcPlan& tp, int nrhs, cudaStream_t s);
// Queue a copy of the flag that a tensor-core pass sets when a bounded wait ran out
// into *host (0 at once where none was launched since the last reading); once the stream has been waited for, tc_err_clear says whether it was set
// and clears it.
void tc_err_async(const TcPlan& tp, int* host, cudaStream_t s);
bool tc_err_clear(const TcPlan& tp, int err, cudaStream_t s);

}  // namespace sldm
