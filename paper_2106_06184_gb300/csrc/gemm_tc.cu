// Complex64 block products with 9 to 32 right-hand sides on the tcgen05 tensor
// cores (the multi-RHS matrix-vector products of GMRES on Eq. finalsystem, one
// pass over the stored blocks per step).
//
// Complex product as one real GEMM.  A complex64 row-major block A (m x n) is,
// byte for byte, a row-major FP32 matrix A' of m rows and 2n columns (re, im
// interleaved).  With B' (2n x 64) holding, for right-hand side r, the columns
//     B'[2c, 2r] = Re x_r[c],  B'[2c+1, 2r] = -Im x_r[c]
//     B'[2c, 2r+1] = Im x_r[c], B'[2c+1, 2r+1] = Re x_r[c],
// D = A' B' holds Re y_r in column 2r and Im y_r in column 2r+1.  A' is the
// stored block itself (the MMA's K-major A operand, streamed by TMA); B' (hi and
// lo, below) is built for every K chunk of every job once per pass by
// tc_bprime_kernel into global memory and streamed by TMA as well (it is the same
// for all row tiles of a job, so building it in each tile would repeat the work).
//
// Near-FP32 accuracy from FP16 operands (three products): every 128-column segment of a
// row of A, and of every column of B', is scaled by a power of two that puts its largest
// entry into [2^14, 2^15) (A's exponents are worked out once with the plan, B''s with
// each pass).  With hi(v) = v rounded to FP16 (11 bits: |v - hi| <= 2^-11 |v|) and lo(v) =
// 2^11 (v - hi) rounded to FP16 (error <= 2^-11 |v - hi| <= 2^-22 |v|; scaled into hi's range, or its last bits
// would fall below FP16's smallest number for small v),
//     D = hi(A) hi(B) + 2^-11 (lo(A) hi(B) + hi(A) lo(B))        (FP32 accumulation of either sum),
// the dropped lo(A) lo(B) (<= 2^-22 |A||B|) and the two roundings of lo leave
// each product term within 3 x 2^-22 of |A||B| (about 2^-22 for typical data),
// against 2^-24 for an FP32 product.  Entries below 2^-29 of their segment's largest keep fewer bits, an
// absolute error of 2^-51 of that largest (TF32 keeps them; FP32 sums of the segment do not).  FP16 has TF32's
// precision at twice its rate and half its bytes: four MMAs per 32 columns instead of
// eight, whose issue (~75 cycles each) bound the TF32 form, and half the B' traffic.  The
// sums are compensated (below).  The TF32 form of the operands (hi and lo rounded to TF32, no
// scales, the same error) is kept for the far field of FP64 operators held as pairs (gemm_tc.h).
//
// Per CTA (one per SM, persistent over its tiles, longest first), 128-row
// tiles streamed in stages of 4 TMA boxes (128 rows x 4 x 128 B, 128-byte
// swizzled): 512 contiguous bytes of every row per stage, which DRAM serves at
// ~0.98 of the copy rate, against ~0.65 for 128-byte runs.  Each stage is
// split into four K sub-chunks of 32 FP32 columns.  Warp-specialised,
// synchronised by mbarriers only:
//   warp 0   TMA: a ring of stages;
//   warp 18  TMA of B' (hi and lo; a box of two sub-chunks, one in TF32) into its shared operand buffers;
//   warps 2-9 split: thread = row, the two warps of 32 rows take the sub-chunks in turn: scaled,
//            rounded to FP16 hi and lo and stored as pairs into one of the TMEM
//            operand buffers (A of tcgen05.mma in tensor memory).  Whole sub-chunks per warp
//            halve the barrier round trips of this chain, which is its length (1,415 -> 1,363 us);
//   warp 1   MMA: one thread issues, per K step of 16 (TF32: 8),
//            hi(A) x [hi(B') | lo(B')] (M 128, N 128: B' hi and lo are the two
//            halves of one 128-row operand) and lo(A) x hi(B') (N 64) into the
//            second half (unscaled TF32: the first), into one of two 128-column TMEM accumulators, a fresh
//            one for every stage (a segment of 128 K columns), and commits them
//            to the operand buffer's barrier;
//   warps 10-17 epilogue: fold each segment's accumulator (the sum of its two
//            halves, scaled back) into compensated FP32 sums in registers (warp w: TMEM
//            lanes 32 (w % 4) .., 32 of the 64 output columns), and at the end
//            of a tile write Y.
// The tensor core rounds its FP32 accumulator at every MMA: a tile's ~10^4
// MMAs into one accumulator would lose ~2^-17 of the result; segments of 16
// MMAs and compensated sums across them keep the product as accurate as an
// FP32 CUDA-core product.
// Tiles are padded to whole stages (zero columns from TMA and zero B').
//
// 8 x 8 metasurface, 32 right-hand sides (6.47 GB): 1,745 us in TF32 -> 1,363 us with unscaled low parts, 1,390 us
// with scaled ones, 0.69 of the HBM copy rate.  The stream of A alone takes 982 us through this ring; the
// rest is the latency of the split and epilogue warps, which share the four schedulers.
#include <cuda.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <queue>
#include <type_traits>

#include <cuda_fp16.h>

#include "gemm_tc.h"
#include "tc_ptx.cuh"

namespace sldm {

namespace {

constexpr int TC_M = 128;
constexpr int TC_N = 2 * TC_MAX_NRHS;  // 64 accumulator columns
constexpr int TC_KC = 32;              // FP32 columns of A per chunk: one 128-byte swizzle row
constexpr int TC_BPS = 4;              // TMA boxes (sub-chunks) per stage
constexpr int TC_R = 2;                // stages in the ring
constexpr int TC_THREADS = 608;        // 19 warps: TMA (A), MMA, 8 split, 8 epilogue, TMA (B')
constexpr int TC_NBB = 6;              // B' operand buffers (shared, hi/lo)
// the two forms of the operands (F: scaled FP16, else TF32)
template <bool F>
struct TcForm {
  static constexpr int AW = F ? 32 : 64;   // TMEM columns of an A operand buffer: hi, lo
  static constexpr int NA = 256 / AW;      // A operand buffers
  static constexpr int BPB = F ? 2 : 1;    // sub-chunks per B' buffer (one box of 128-byte rows)
  static constexpr int KS = F ? 16 : 8;    // K of an MMA
};
constexpr uint32_t TC_A_BYTES = TC_M * TC_KC * 4;  // 16 KB: one box, one sub-chunk
constexpr uint32_t TC_STAGE_BYTES = TC_BPS * TC_A_BYTES;
constexpr int TC_BK = 2 * TC_KC;                    // K columns of a B' box in FP16: one 128-byte swizzle row
constexpr uint32_t TC_B_BYTES = TC_N * 128;         // 8 KB
constexpr uint32_t TC_BBUF = 2 * TC_B_BYTES;       // B' hi, lo
constexpr uint32_t TC_RING = TC_R * TC_STAGE_BYTES;
// TMEM: two accumulators of 128 columns (hi(A) hi(B') in 0-63, hi(A) lo(B') + lo(A) hi(B') in
// 64-127; TF32: lo(A) hi(B') in 0-63) at columns 0 and 128, A operand buffers (hi and lo: 16 columns of FP16 pairs or 32 of TF32 each) from 256
constexpr uint32_t TC_TMEM_COLS = 512;
constexpr uint32_t TC_ACC_COLS = 2 * TC_N;
constexpr uint32_t TC_ACC_COL = 0, TC_AOP_COL = 2 * TC_ACC_COLS;
static_assert(TC_AOP_COL + 256 <= TC_TMEM_COLS, "accumulators and operand buffers exceed the TMEM allocation");
constexpr int TC_NBARS = 2 * TC_R + 2 * 8 + 4 + 2 * TC_NBB;
constexpr size_t TC_BAR_BYTES = 512;
constexpr size_t TC_SMEM = size_t(TC_RING) + TC_NBB * size_t(TC_BBUF) + 1024 + TC_BAR_BYTES;
static_assert(8 * TC_NBARS + 4 <= TC_BAR_BYTES, "barriers and the TMEM slot exceed their shared-memory space");

static_assert(TC_BBUF % 1024 == 0 && TC_A_BYTES % 1024 == 0 && TC_B_BYTES % 1024 == 0, "swizzle atoms are 1 KB aligned");
static_assert(TC_SMEM <= 227 * 1024, "ring and operand buffers exceed the shared memory of a CTA");

// instruction descriptor: D FP32 (bits 4-5 = 1), A and B FP16 or TF32 (bits
// 7-9, 10-12 = 0 or 2), both K-major (bits 15, 16 = 0), N >> 3 at bits 17-22, M >> 4 at 24-28
__host__ __device__ constexpr uint32_t tc_idesc(bool f16, int n) {
  return (1u << 4) | (f16 ? 0u : (2u << 7) | (2u << 10)) | (uint32_t(n >> 3) << 17) | (uint32_t(TC_M >> 4) << 24);
}

// D (TMEM) (+)= A (TMEM: lane = row, one TF32 per column) x B (shared memory descriptor)
__device__ __forceinline__ void tc_mma_tf32(uint32_t d_tmem, uint32_t a_tmem, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// 8 consecutive accumulator columns of this warp's 32 TMEM lanes, at two column offsets
__device__ __forceinline__ void tmem_ld8x2(uint32_t taddr, uint32_t off, f2 (&v)[4], f2 (&w)[4]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%16];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8, %9, %10, %11, %12, %13, %14, %15}, [%17];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr), "r"(taddr + off)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[i] = f2_pack(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
    w[i] = f2_pack(__uint_as_float(r[8 + 2 * i]), __uint_as_float(r[9 + 2 * i]));
  }
}
// 8 consecutive TMEM columns of this warp's 32 lanes from registers
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// FP32 -> TF32 (10 mantissa bits), round to nearest, ties away from zero: the
// result is an FP32 value with its 13 low mantissa bits zero, which the MMA
// takes exactly.  On the bit pattern: add half of the dropped unit (0x1000,
// carrying into the exponent when the mantissa overflows) and clear the 13
// bits - two full-rate integer operations (finite inputs below ~3.4e38)
__device__ __forceinline__ float tf32_rn(float v) {
  return __uint_as_float((__float_as_uint(v) + 0x1000u) & 0xFFFFE000u);
}
// v = hi + lo: hi = tf32(v) (|v - hi| <= 2^-11 |v|), lo = tf32(v - hi) (rounding
// error <= 2^-11 |v - hi| <= 2^-22 |v|), both exact TF32 operands
__device__ __forceinline__ void tf32_split(float v, float& hi, float& lo) {
  hi = tf32_rn(v);
  lo = tf32_rn(v - hi);
}
// 16 consecutive TMEM columns of this warp's 32 lanes from registers
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16};\n" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
      "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
      "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
      : "memory");
}
// v = hi + 2^-11 lo, both FP16 pairs (the first number in the lower half), rounded to nearest
constexpr float LO_UP = 0x1p11f, LO_DOWN = 0x1p-11f;
__device__ __forceinline__ void f16_split(f2 v, uint32_t& hi, uint32_t& lo) {
  float a, b;
  f2_unpack(v, a, b);
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  f2_unpack(f2_mul(f2_sub(v, f2_pack(f.x, f.y)), f2_pack(LO_UP, LO_UP)), a, b);
  const __half2 l = __floats2half2_rn(a, b);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
}  // namespace

// 19 warps over the 4 SM sub-partitions (5, 5, 5, 4) x 32 threads x 96 registers <= 16,384 each
template <bool F>
__global__ void __maxnreg__(96)
    gemm_tc_kernel(const GemvJob* __restrict__ jobs, const unsigned char* __restrict__ maps, const TcTile* __restrict__ tiles,
                   const int32_t* __restrict__ cta_begin, const unsigned char* __restrict__ bmap,
                   const TcJob* __restrict__ tj, const signed char* __restrict__ aexp, const float* __restrict__ bscale,
                   int nrhs, int* err) {
  constexpr int TC_NA = TcForm<F>::NA, AW = TcForm<F>::AW, BPB = TcForm<F>::BPB, KS = TcForm<F>::KS;
  constexpr uint32_t IDESC_N64 = tc_idesc(F, TC_N), IDESC_N128 = tc_idesc(F, 2 * TC_N);
  extern __shared__ unsigned char tc_raw[];
  const int t_begin = cta_begin[blockIdx.x], t_end = cta_begin[blockIdx.x + 1];
  if (t_begin >= t_end) return;
  const uint32_t raw = smem_u32(tc_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;  // ring[R], B'[NB]
  unsigned char* gb = tc_raw + (base - raw);
  const uint32_t bbuf0 = base + TC_RING;
  const uint32_t bars = bbuf0 + TC_NBB * TC_BBUF;
  // barriers (8 bytes each): full[R], empty[R], ready[NA], wfree[NA], accfull[2], accempty[2], bfull[NBB], bfree[NBB]
  auto full = [&](int s) { return bars + 8u * uint32_t(s); };
  auto empty = [&](int s) { return bars + 8u * uint32_t(TC_R + s); };
  auto ready = [&](int b) { return bars + 8u * uint32_t(2 * TC_R + b); };
  auto wfree = [&](int b) { return bars + 8u * uint32_t(2 * TC_R + TC_NA + b); };
  auto accfull = [&](int a) { return bars + 8u * uint32_t(2 * TC_R + 2 * TC_NA + a); };
  auto accempty = [&](int a) { return bars + 8u * uint32_t(2 * TC_R + 2 * TC_NA + 2 + a); };
  auto bfull = [&](int b) { return bars + 8u * uint32_t(2 * TC_R + 2 * TC_NA + 4 + b); };
  auto bfree = [&](int b) { return bars + 8u * uint32_t(2 * TC_R + 2 * TC_NA + 4 + TC_NBB + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gb + (bars - base) + 8 * TC_NBARS);
  __shared__ int s_fail;
  volatile int* vfail = &s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int q = 0; q < TC_R; ++q) {
      mbar_init(full(q), 1);
      mbar_init(empty(q), 8);
    }
    for (int b = 0; b < TC_NA; ++b) {
      mbar_init(ready(b), 4);
      mbar_init(wfree(b), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(accfull(a), 1);
      mbar_init(accempty(a), 8);
    }
    for (int b = 0; b < TC_NBB; ++b) {
      mbar_init(bfull(b), 1);
      mbar_init(bfree(b), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TC_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // sub-chunks of a tile, padded to whole stages
  auto nk_of = [&](int t) { return tiles[t].nk; };
  int total = 0;  // sub-chunks of this CTA (a multiple of TC_BPS)
  for (int t = t_begin; t < t_end; ++t) total += nk_of(t);
  const int nstages = total / TC_BPS;

  if (warp == 0) {
    // ---------------- TMA producer: one stage = 4 boxes along K
    if (lane == 0) {
      int tile = t_begin, k = 0, nk = nk_of(t_begin), st = 0;
      for (; st < nstages; ++st) {
        const int q = st % TC_R;
        if (st >= TC_R && !mbar_wait(empty(q), uint32_t(((st / TC_R) - 1) & 1), vfail)) {
          *vfail = 1;
          break;
        }
        const TcTile T = tiles[tile];
        mbar_expect_tx(full(q), TC_STAGE_BYTES);
#pragma unroll
        for (int bx = 0; bx < TC_BPS; ++bx)
          tma_load_2d(base + uint32_t(q) * TC_STAGE_BYTES + uint32_t(bx) * TC_A_BYTES, maps + size_t(T.job) * 128,
                      (T.k0 + k + bx) * TC_KC, T.row0, full(q));
        k += TC_BPS;
        if (k == nk) {
          k = 0;
          if (++tile < t_end) nk = nk_of(tile);
        }
      }
      // the loads in flight (the latest stage of each slot) land before the CTA leaves
      for (int q = (st > TC_R ? st - TC_R : 0); q < st; ++q) mbar_wait(full(q % TC_R), uint32_t((q / TC_R) & 1));
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int tile_i = 0, k = 0, nk = nk_of(t_begin), last = -1;
      for (int g = 0; g < total; ++g) {
        const int b = g % TC_NA, gb = g / BPB, bb = gb % TC_NBB, seg = g / TC_BPS, j = g % TC_BPS;
        bool ok = true;
        if (j == 0 && seg >= 2) ok = mbar_wait(accempty(seg & 1), uint32_t(((seg >> 1) - 1) & 1), vfail);
        if (ok && g % BPB == 0) ok = mbar_wait(bfull(bb), uint32_t((gb / TC_NBB) & 1), vfail);
        if (ok) ok = mbar_wait(ready(b), uint32_t((g / TC_NA) & 1), vfail);
        if (!ok) {
          *vfail = 1;
          break;
        }
        tc_fence_after();
        const uint32_t acc = tmem + TC_ACC_COL + uint32_t(seg & 1) * TC_ACC_COLS;
        const uint32_t aop = tmem + TC_AOP_COL + uint32_t(b) * AW;  // hi, then lo
        // B' hi rows 0-63, lo rows 64-127; this sub-chunk's half of the 128-byte rows
        const uint32_t bh = bbuf0 + uint32_t(bb) * TC_BBUF + uint32_t(g % BPB) * 64u;
#pragma unroll
        for (int ks = 0; ks < TC_KC / KS; ++ks) {
          const uint32_t o = uint32_t(ks) * 32u;  // 16 FP16 or 8 TF32 = 32 bytes along K in the swizzle row of B'
          const uint32_t ac = uint32_t(ks) * 8u;  // 8 TMEM columns of A
          const uint32_t acc0 = (j > 0 || ks > 0) ? 1u : 0u;  // a fresh accumulator per segment
          // hi(A) [hi(B') | lo(B')] in one N = 128 product, then lo(A) hi(B') into columns 64-127 (TF32: 0-63)
          if constexpr (F) {
            tc_mma_f16(acc, aop + ac, sw128_desc(bh + o), IDESC_N128, acc0);
            tc_mma_f16(acc + TC_N, aop + AW / 2 + ac, sw128_desc(bh + o), IDESC_N64, 1u);
          } else {
            tc_mma_tf32(acc, aop + ac, sw128_desc(bh + o), IDESC_N128, acc0);
            tc_mma_tf32(acc, aop + AW / 2 + ac, sw128_desc(bh + o), IDESC_N64, 1u);
          }
        }
        tc_commit(wfree(b));
        if (g % BPB == BPB - 1) tc_commit(bfree(bb));
        if (j == TC_BPS - 1) tc_commit(accfull(seg & 1));
        last = g;
        if (++k == nk) {
          k = 0;
          ++tile_i;
          if (t_begin + tile_i < t_end) nk = nk_of(t_begin + tile_i);
        }
      }
      // the MMAs in flight (they complete in order) finish, and their commits arrive, before the CTA leaves
      if (last >= 0) {
        mbar_wait(wfree(last % TC_NA), uint32_t((last / TC_NA) & 1));
        if (last % BPB == BPB - 1) mbar_wait(bfree(last / BPB % TC_NBB), uint32_t((last / BPB / TC_NBB) & 1));
        if (last % TC_BPS == TC_BPS - 1) mbar_wait(accfull(last / TC_BPS & 1), uint32_t((last / TC_BPS >> 1) & 1));
      }
    }
    __syncwarp();
  } else if (warp < 10) {
    // ---------------- split warps: thread = row of the tile (TMEM lane quarter warp % 4); the
    // two warps of a lane quarter take the sub-chunks in turn
    const int q4 = warp & 3, kh = (warp - 2) >> 2, row = 32 * q4 + lane;
    // scale exponents of this row, one stage ahead of their use
    int tile = t_begin, k = 0, nk = 0, mpad = 0;
    const signed char* ea = nullptr;
    auto next_exp = [&]() {
      if (k == nk) {
        if (tile == t_end) return 0;
        const TcTile T = tiles[tile++];
        const TcJob J = tj[T.job];
        k = 0;
        nk = T.nk;
        mpad = J.mpad;
        ea = aexp + J.aexp + int64_t(T.k0 / TC_BPS) * mpad + T.row0 + row;
      }
      const int e = *ea;
      ea += mpad;
      k += TC_BPS;
      return e;
    };
    int enext = F ? next_exp() : 0;
    f2 sc2 = f2_pack(1.f, 1.f);
    for (int g = kh; g < total; g += 2) {
      const int st = g / TC_BPS, j = g % TC_BPS, q = st % TC_R, b = g % TC_NA;
      if (F && j == kh) {  // this row's scale for the stage
        sc2 = f2_pack(pow2f(enext), pow2f(enext));
        enext = next_exp();
      }
      bool ok = mbar_wait(full(q), uint32_t((st / TC_R) & 1), vfail);
      if (ok && g >= TC_NA) ok = mbar_wait(wfree(b), uint32_t(((g / TC_NA) - 1) & 1), vfail);
      ok = __all_sync(0xffffffffu, ok);  // the TMEM stores below need the whole warp
      if (!ok) {
        *vfail = 1;
        break;
      }
      // this row of box j of the landed stage: 8 x 16 B, swizzled
      const unsigned char* rp = gb + size_t(q) * TC_STAGE_BYTES + size_t(j) * TC_A_BYTES + size_t(row) * 128;
      const uint32_t ta = tmem + (uint32_t(32 * q4) << 16) + TC_AOP_COL + uint32_t(b) * AW;
      float4 a[8];
#pragma unroll
      for (int jj = 0; jj < 8; ++jj) a[jj] = *reinterpret_cast<const float4*>(rp + ((jj ^ (row & 7)) * 16));
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        if constexpr (!F) {
          float h[16], l[16];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const float4 v = a[4 * hf + jj];
            tf32_split(v.x, h[4 * jj], l[4 * jj]);
            tf32_split(v.y, h[4 * jj + 1], l[4 * jj + 1]);
            tf32_split(v.z, h[4 * jj + 2], l[4 * jj + 2]);
            tf32_split(v.w, h[4 * jj + 3], l[4 * jj + 3]);
          }
          tmem_st16(ta + uint32_t(16 * hf), h);
          tmem_st16(ta + AW / 2 + uint32_t(16 * hf), l);
          continue;
        }
        uint32_t h[8], l[8];
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const float4 v = a[4 * hf + jj];
          f16_split(f2_mul(f2_pack(v.x, v.y), sc2), h[2 * jj], l[2 * jj]);
          f16_split(f2_mul(f2_pack(v.z, v.w), sc2), h[2 * jj + 1], l[2 * jj + 1]);
        }
        tmem_st8(ta + uint32_t(8 * hf), h);
        tmem_st8(ta + AW / 2 + uint32_t(8 * hf), l);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (j >= TC_BPS - 2) mbar_arrive(empty(q));  // this warp's last sub-chunk of the stage
        mbar_arrive(ready(b));                        // A of this sub-chunk is in TMEM
      }
    }
  } else if (warp == 18) {
    // ---------------- TMA producer of B' (hi rows 0-63, lo rows 64-127 of one box per two
    // sub-chunks, built for the pass by tc_bprime_kernel) into the operand buffers
    if (lane == 0) {
      int tile = t_begin, k = 0, nk = nk_of(t_begin), g = 0;
      for (; g < total / BPB; ++g) {
        const int b = g % TC_NBB;
        if (g >= TC_NBB && !mbar_wait(bfree(b), uint32_t(((g / TC_NBB) - 1) & 1), vfail)) {
          *vfail = 1;
          break;
        }
        mbar_expect_tx(bfull(b), TC_BBUF);
        tma_load_2d(bbuf0 + uint32_t(b) * TC_BBUF, bmap, 0, 2 * TC_N * (tj[tiles[tile].job].base * (2 / BPB) + (tiles[tile].k0 + k) / BPB),
                    bfull(b));
        if ((k += BPB) == nk) {
          k = 0;
          if (++tile < t_end) nk = nk_of(tile);
        }
      }
      // the loads in flight land before the CTA leaves
      for (int q = (g > TC_NBB ? g - TC_NBB : 0); q < g; ++q) mbar_wait(bfull(q % TC_NBB), uint32_t((q / TC_NBB) & 1));
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps: TMEM lane quarter warp % 4, accumulator columns 32 half ..
    const int q4 = warp & 3, half = (warp - 10) >> 2;
    // compensated sums of this row's 32 columns over the tile's segments, as the pairs
    // (re, im) of 16 right-hand sides: packed FP32 operations, half the issue slots (these warps and
    // the split warps share them; with single ones this kernel was bound there)
    f2 cs[16], cc[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) cs[i] = cc[i] = 0ull;
    int seg = 0;
    for (int t = t_begin; t < t_end; ++t) {
      const int nseg = nk_of(t) / TC_BPS;
      bool ok = true;
      // the scales of the tile's segments: this row's of A, and in lane i the one of right-hand side 16 half + i
      const signed char* ea;
      const float* eb;
      int mpad;
      {
        const TcTile T = tiles[t];
        const TcJob TJ = tj[T.job];
        mpad = TJ.mpad;
        ea = aexp + TJ.aexp + int64_t(T.k0 / TC_BPS) * mpad + T.row0 + 32 * q4 + lane;
        eb = bscale + (TJ.base / 2 + T.k0 / TC_BPS) * TC_MAX_NRHS + half * 16 + (lane & 15);
      }
      for (int sg = 0; sg < nseg; ++sg, ++seg) {
        float sa = 1.f, sbl = 1.f;
        if (F) {  // before the wait for the segment
          sa = pow2f(-*ea);
          sbl = __ldg(eb);
          ea += mpad;
          eb += TC_MAX_NRHS;
        }
        ok = __all_sync(0xffffffffu, mbar_wait(accfull(seg & 1), uint32_t((seg >> 1) & 1), vfail));
        if (!ok) break;  // the TMEM loads below need the whole warp
        tc_fence_after();
#pragma unroll
        for (int hq = 0; hq < 4; ++hq) {
          f2 v[4], w[4];  // hi(A) hi(B'), and hi(A) lo(B') + lo(A) hi(B') (TF32: lo(A) hi(B') in the first)
          tmem_ld8x2(tmem + (uint32_t(32 * q4) << 16) + TC_ACC_COL + uint32_t(seg & 1) * TC_ACC_COLS +
                         uint32_t(half * 32 + 8 * hq),
                     TC_N, v, w);
#pragma unroll
          for (int i = 0; i < 4; ++i) {  // 8 columns = 4 right-hand sides
            const int c = 4 * hq + i;
            f2 u = F ? f2_fma(w[i], f2_pack(LO_DOWN, LO_DOWN), v[i]) : f2_add(v[i], w[i]);
            if (F) {
              const float sb = __shfl_sync(0xffffffffu, sbl, c);
              u = f2_mul(f2_mul(u, f2_pack(sa, sa)), f2_pack(sb, sb));
            }
            // TwoSum (Knuth): cs + cc carries the running sum
            const f2 sum = f2_add(cs[c], u), bp = f2_sub(sum, cs[c]);
            cc[c] = f2_add(cc[c], f2_add(f2_sub(cs[c], f2_sub(sum, bp)), f2_sub(u, bp)));
            cs[c] = sum;
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accempty(seg & 1));  // the accumulator may take the next segment
      }
      if (!ok) {
        *vfail = 1;
        break;
      }
      const TcTile T = tiles[t];
      const GemvJob& J = jobs[T.job];
      const int row = T.row0 + 32 * q4 + lane;
      if (row < J.m) {
        float2* y = reinterpret_cast<float2*>(J.y);
        const float ar = float(J.ar), ai = float(J.ai);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const int r = half * 16 + c;
          if (r < nrhs) {
            float re, im;
            f2_unpack(f2_add(cs[c], cc[c]), re, im);
            float2 o = make_float2(ar * re - ai * im, ar * im + ai * re);
            float2* yy = y + int64_t(r) * J.ldy + row;
            if (T.split) {
              atomicAdd(yy, o);  // one of the two K halves of the tile (Y zeroed before the pass)
            } else {
              if (J.beta) {
                const float2 bb = *yy;
                o.x += bb.x;
                o.y += bb.y;
              }
              *yy = o;
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) cs[i] = cc[i] = 0ull;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && *vfail) atomicExch(err, 1);
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
}

// B' of one stage (64 complex columns, two boxes of 64 K columns) per block: for
// right-hand side r and complex column c row 2r holds (Re x_r[c], -Im x_r[c]) and row 2r + 1
// (Im x_r[c], Re x_r[c]) at K columns 2c, 2c + 1, scaled by the power of two of the right-hand
// side's largest entry in the stage, FP16 hi (rows 0-63) and lo (64-127) parts, row-major (TMA
// applies the 128-byte swizzle); zero for r >= nrhs and beyond the job's columns.
// bscale[stage][r] undoes the scale.  8 threads per right-hand side, 8 columns each.
// Blocks nstage and above zero the Y rows of the tiles split along K.
__global__ void __launch_bounds__(256) tc_bprime_kernel(const GemvJob* __restrict__ jobs, const int32_t* __restrict__ gjob,
                                                        const int32_t* __restrict__ gst, int nstage,
                                                        const TcTile* __restrict__ ztiles, int nrhs, __half* __restrict__ bp,
                                                        float* __restrict__ bscale) {
  const int gidx = blockIdx.x;
  if (gidx >= nstage) {  // Y rows of a tile split along K: zeroed, the two halves add into them
    const TcTile T = ztiles[gidx - nstage];
    const GemvJob& J = jobs[T.job];
    float2* y = reinterpret_cast<float2*>(J.y);
    for (int e = threadIdx.x; e < TC_M * nrhs; e += blockDim.x) {
      const int row = T.row0 + e % TC_M, r = e / TC_M;
      if (row < J.m) y[int64_t(r) * J.ldy + row] = make_float2(0.f, 0.f);
    }
    return;
  }
  const GemvJob& J = jobs[gjob[gidx]];
  const int r = threadIdx.x >> 3, sub = threadIdx.x & 7;
  const int c0 = gst[gidx] * (2 * TC_KC) + sub * 8;  // 64 complex columns per stage
  const float2* x = reinterpret_cast<const float2*>(J.x) + int64_t(r) * J.ldx;
  float2 v[8];
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    v[i] = r < nrhs && c0 + i < J.n ? x[c0 + i] : make_float2(0.f, 0.f);
    m = fmaxf(m, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
  }
  for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = tc_scale_exp(m);
  const float sc = pow2f(e);
  if (sub == 0) bscale[int64_t(gidx) * TC_MAX_NRHS + r] = pow2f(-e);
  uint32_t h0[8], l0[8], h1[8], l1[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float re = sc * v[i].x, im = sc * v[i].y;
    f16_split(f2_pack(re, -im), h0[i], l0[i]);
    f16_split(f2_pack(im, re), h1[i], l1[i]);
  }
  // box 2 gidx + (sub / 4), row, 8 pairs from K column 16 (sub % 4)
  __half* box = bp + (size_t(2 * gidx + (sub >> 2)) * 2 * TC_N) * TC_BK + 16 * (sub & 3);
  auto put = [&](int row, const uint32_t (&w)[8]) {
    uint4* d = reinterpret_cast<uint4*>(box + size_t(row) * TC_BK);
    d[0] = make_uint4(w[0], w[1], w[2], w[3]);
    d[1] = make_uint4(w[4], w[5], w[6], w[7]);
  };
  put(2 * r, h0);
  put(2 * r + 1, h1);
  put(TC_N + 2 * r, l0);
  put(TC_N + 2 * r + 1, l1);
}

// Scale exponents of A: one per row and stage (128 FP32 columns = 512 bytes of the row),
// one warp each; aexp[stage][row] per job (blockIdx.y), rows padded to whole tiles.
__global__ void __launch_bounds__(256) tc_aexp_kernel(const GemvJob* __restrict__ jobs, const TcJob* __restrict__ tj, int job0,
                                                      signed char* __restrict__ aexp) {
  const GemvJob& J = jobs[job0 + blockIdx.y];
  const TcJob T = tj[job0 + blockIdx.y];
  const int lane = threadIdx.x & 31, nst = (2 * J.n + TC_KC * TC_BPS - 1) / (TC_KC * TC_BPS);
  const int64_t total = int64_t(J.m) * nst;
  for (int64_t w = (int64_t(blockIdx.x) * 256 + threadIdx.x) >> 5; w < total; w += int64_t(gridDim.x) * 8) {
    const int64_t row = w / nst;
    const int st = int(w % nst);
    const float2* a = reinterpret_cast<const float2*>(J.A) + row * J.lda;
    float m = 0.f;
    for (int c = st * (TC_KC * TC_BPS / 2) + lane, i = 0; i < 2; ++i, c += 32)
      if (c < J.n) {
        const float2 v = a[c];
        m = fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y)));
      }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) aexp[T.aexp + int64_t(st) * T.mpad + row] = static_cast<signed char>(tc_scale_exp(m));
  }
}

// B' of every sub-chunk of the pass (hi rows 0-63, lo rows 64-127, 32 FP32 columns
// each, row-major; TMA applies the 128-byte swizzle): for right-hand side r and
// complex column c = 16 kc + u / 2 of the sub-chunk's job, row 2r holds
// (Re x_r[c], -Im x_r[c]) and row 2r + 1 (Im x_r[c], Re x_r[c]) at columns u, u + 1
// (u even), TF32 hi and lo parts; zero for r >= nrhs and beyond the job's columns.
// Blocks nsub and above zero the Y rows of the tiles split along K.
__global__ void tf32_bprime_kernel(const GemvJob* __restrict__ jobs, const int32_t* __restrict__ gjob,
                                 const int32_t* __restrict__ gst, int nsub, const TcTile* __restrict__ ztiles, int nrhs,
                                 float* __restrict__ bp) {
  const int gidx = blockIdx.x;
  if (gidx >= nsub) {  // Y rows of a tile split along K: zeroed, the two halves add into them
    const TcTile T = ztiles[gidx - nsub];
    const GemvJob& J = jobs[T.job];
    float2* y = reinterpret_cast<float2*>(J.y);
    for (int e = threadIdx.x; e < TC_M * nrhs; e += blockDim.x) {
      const int row = T.row0 + e % TC_M, r = e / TC_M;
      if (row < J.m) y[int64_t(r) * J.ldy + row] = make_float2(0.f, 0.f);
    }
    return;
  }
  const GemvJob& J = jobs[gjob[gidx / TC_BPS]];
  const int kc = gst[gidx / TC_BPS] * TC_BPS + gidx % TC_BPS;
  const float2* x = reinterpret_cast<const float2*>(J.x);
  for (int e = threadIdx.x; e < TC_N * TC_KC / 2; e += blockDim.x) {  // (row, complex column) pairs
    const int brow = e / (TC_KC / 2), cl = e % (TC_KC / 2);
    const int r = brow >> 1, c = kc * (TC_KC / 2) + cl;
    float2 v = make_float2(0.f, 0.f);
    if (r < nrhs && c < J.n) v = x[int64_t(r) * J.ldx + c];
    const float a0 = (brow & 1) ? v.y : v.x, a1 = (brow & 1) ? v.x : -v.y;
    float h0, l0, h1, l1;
    tf32_split(a0, h0, l0);
    tf32_split(a1, h1, l1);
    float* hi = bp + (size_t(gidx) * 2 * TC_N + brow) * TC_KC + 2 * cl;
    float* lo = hi + size_t(TC_N) * TC_KC;
    *reinterpret_cast<float2*>(hi) = make_float2(h0, h1);
    *reinterpret_cast<float2*>(lo) = make_float2(l0, l1);
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encoder() {
  // looked up once (thread-safe initialisation of a local static)
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    return EncodeTiledFn(nullptr);
  }();
  return fn;
}

bool tc_map_2d(int type, const void* p, uint64_t nx, uint64_t ny, uint64_t pitch, int bx, int by, unsigned char* out) {
  static_assert(sizeof(CUtensorMap) == 128, "tensor map size");
  const EncodeTiledFn enc = encoder();
  if (!enc || pitch % 16 != 0 || (reinterpret_cast<uintptr_t>(p) & 15) != 0) return false;
  alignas(64) CUtensorMap map;
  const cuuint64_t dims[2] = {nx, ny};
  const cuuint64_t strides[1] = {pitch};
  const cuuint32_t box[2] = {cuuint32_t(bx), cuuint32_t(by)};
  const cuuint32_t estr[2] = {1, 1};
  if (enc(&map, CUtensorMapDataType(type), 2, const_cast<void*>(p), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  std::memcpy(out, &map, 128);
  return true;
}
bool tc_block_map(const void* A, int64_t lda, int m, int n, unsigned char* out) {
  return m > 0 && n > 0 && tc_map_2d(CU_TENSOR_MAP_DATA_TYPE_FLOAT32, A, uint64_t(2) * n, m, uint64_t(lda) * 8, TC_KC, TC_M, out);
}

void tc_plan_build(const std::vector<GemvJob>& jobs, TcPlan& tp, bool f16, cudaStream_t s) {
  tp.ok = false;
  tp.f16 = f16;
  tp.longest = 0;
  if (jobs.empty()) return;
  std::vector<unsigned char> maps(jobs.size() * 128);
  std::vector<TcTile> tl;
  std::vector<int> cost;
  std::vector<int32_t> gjob, gst;
  std::vector<TcJob> tjobs;
  int64_t aexp_n = 0;
  std::vector<TcTile> tp_zero;  // tiles split along K: their Y rows are zeroed before each pass
  for (size_t i = 0; i < jobs.size(); ++i) {
    const GemvJob& J = jobs[i];
    if (!tc_block_map(J.A, J.lda, J.m, J.n, &maps[i * 128])) return;
    const int nk = ((2 * J.n + TC_KC - 1) / TC_KC + TC_BPS - 1) / TC_BPS * TC_BPS;
    const int nst = nk / TC_BPS, mpad = (J.m + TC_M - 1) / TC_M * TC_M;
    tjobs.push_back({aexp_n, mpad, 2 * int32_t(gjob.size())});
    aexp_n += int64_t(nst) * mpad;
    for (int st = 0; st < nst; ++st) {
      gjob.push_back(int32_t(i));
      gst.push_back(st);
    }
    for (int r0 = 0; r0 < J.m; r0 += TC_M) {
      tl.push_back({int32_t(i), r0, 0, nk, 0});
      cost.push_back(nk);
    }
  }
  int dev = 0, nsm = 0;
  SLDM_CUDA(cudaGetDevice(&dev));
  SLDM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // Tiles are whole rows of 128 x the job's K: a few long tiles against the SM
  // count leave CTAs idle at the end (the longest-first assignment of 180 tiles
  // of one length to 152 CTAs gives 28 of them two).  Tiles longer than 0.3 of
  // a CTA's mean load are split into two K halves (whole stages) that add into
  // Y atomically: two additions into zero commute, so the result stays
  // independent of their order.  Jobs that accumulate into Y (beta) keep whole tiles.
  {
    long long tot = 0;
    for (int c : cost) tot += c;
    const double lim = 0.3 * double(tot) / double(std::max(1, std::min<int>(nsm, int(tl.size()))));
    const size_t n0 = tl.size();
    for (size_t i = 0; i < n0; ++i) {
      if (cost[i] < 4 * TC_BPS || double(cost[i]) <= lim || jobs[tl[i].job].beta) continue;
      const int h = cost[i] / TC_BPS / 2 * TC_BPS;
      TcTile b = tl[i];
      b.k0 = h;
      b.nk = cost[i] - h;
      b.split = 1;
      tl[i].nk = h;
      tl[i].split = 1;
      cost[i] = h;
      tp_zero.push_back(tl[i]);
      tl.push_back(b);
      cost.push_back(b.nk);
    }
  }
  // longest tiles first, each to the least loaded CTA
  const int nctas = std::max(1, std::min<int>(nsm, int(tl.size())));
  std::vector<size_t> order(tl.size());
  for (size_t i = 0; i < order.size(); ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](size_t a, size_t b) { return cost[a] > cost[b]; });
  std::vector<std::vector<TcTile>> per(nctas);
  typedef std::pair<long long, int> LoadCta;
  std::priority_queue<LoadCta, std::vector<LoadCta>, std::greater<LoadCta>> pq;
  for (int c = 0; c < nctas; ++c) pq.push({0, c});
  for (size_t i : order) {
    LoadCta lc = pq.top();
    pq.pop();
    per[lc.second].push_back(tl[i]);
    pq.push({lc.first + cost[i], lc.second});
    tp.longest = std::max(tp.longest, int((lc.first + cost[i]) / TC_BPS));
  }
  std::vector<TcTile> flat;
  std::vector<int32_t> begin(1, 0);
  for (auto& v : per) {
    flat.insert(flat.end(), v.begin(), v.end());
    begin.push_back(int32_t(flat.size()));
  }
  // B' for every stage and its tensor map (boxes of 128 rows x 128 B, swizzled like the A boxes)
  tp.nstage = int(gjob.size());
  const uint64_t brows = uint64_t(tp.nstage) * (f16 ? 2 : 4) * 2 * TC_N;  // of 128 bytes
  tp.bprime.alloc(size_t(brows) * 128);
  tp.bscale.alloc(size_t(tp.nstage) * TC_MAX_NRHS);
  std::vector<unsigned char> bmv(128);
  const int bx = f16 ? TC_BK : TC_KC;
  if (!tc_map_2d(f16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, tp.bprime.p, bx, brows, 128, bx, 2 * TC_N,
                 bmv.data()))
    return;
  tp.bmap.upload(bmv, s);
  tp.nzero = int(tp_zero.size());
  if (tp.nzero > 0) tp.ztiles.upload(tp_zero, s);
  tp.tj.upload(tjobs, s);
  tp.gjob.upload(gjob, s);
  tp.gst.upload(gst, s);
  tp.aexp.alloc(size_t(aexp_n));
  tp.aexp.zero(s);
  {
    DBuf<GemvJob> dj;
    dj.upload(jobs, s);
    for (size_t i = 0; i < jobs.size(); i += 65535)  // two waves of CTAs per job: small jobs leave most of theirs idle
      tc_aexp_kernel<<<dim3(152 * 16, unsigned(std::min<size_t>(65535, jobs.size() - i))), 256, 0, s>>>(dj.p, tp.tj.p, int(i),
                                                                                                  tp.aexp.p),
          count_launch();
    SLDM_CUDA(cudaGetLastError());
    SLDM_CUDA(cudaStreamSynchronize(s));
  }
  tp.maps.upload(maps, s);
  tp.tiles.upload(flat, s);
  tp.cta_begin.upload(begin, s);
  tp.err.alloc(1);
  tp.err.zero(s);
  tp.nctas = nctas;
  SLDM_CUDA(cudaStreamSynchronize(s));
  tp.ok = true;
}

void gemm_tc(const GemvPlan& plan, const TcPlan& tp, int nrhs, cudaStream_t s) {
  SLDM_REQUIRE(tp.ok && nrhs >= 1 && nrhs <= TC_MAX_NRHS, SLDM_EINVAL, "tensor-core product: invalid plan or nrhs");
  static std::atomic<uint64_t> attr_set{0};  // devices whose attributes are set
  int dev = 0;
  SLDM_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (!(attr_set.load() & bit)) {
    SLDM_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(TC_SMEM)));
    SLDM_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(TC_SMEM)));
    attr_set.fetch_or(bit);
  }
  ScopedTimer tm("gemm_tc", s);
  auto go = [&](auto f) {
    gemm_tc_kernel<decltype(f)::value><<<unsigned(tp.nctas), TC_THREADS, TC_SMEM, s>>>(plan.jobs, tp.maps.p, tp.tiles.p, tp.cta_begin.p,
                                                                                       tp.bmap.p, tp.tj.p, tp.aexp.p, tp.bscale.p, nrhs,
                                                                                       tp.err.p);
    count_launch();
  };
  if (tp.f16) {
    tc_bprime_kernel<<<unsigned(tp.nstage + tp.nzero), 256, 0, s>>>(plan.jobs, tp.gjob.p, tp.gst.p, tp.nstage, tp.ztiles.p, nrhs,
                                                                    reinterpret_cast<__half*>(tp.bprime.p), tp.bscale.p);
    count_launch();
    go(std::true_type{});
  } else {
    const int nsub = tp.nstage * TC_BPS;
    tf32_bprime_kernel<<<unsigned(nsub + tp.nzero), 256, 0, s>>>(plan.jobs, tp.gjob.p, tp.gst.p, nsub, tp.ztiles.p, nrhs,
                                                                 reinterpret_cast<float*>(tp.bprime.p));
    count_launch();
    go(std::false_type{});
  }
  SLDM_CUDA(cudaGetLastError());
  tp.ran = true;
  if (take_tc_wait()) SLDM_CUDA(cudaMemsetAsync(tp.err.p, 1, sizeof(int), s));
}

void tc_err_async(const TcPlan& tp, int* host, cudaStream_t s) {
  *host = 0;
  if (tp.ran) SLDM_CUDA(cudaMemcpyAsync(host, tp.err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  tp.ran = false;
}
bool tc_err_clear(const TcPlan& tp, int err, cudaStream_t s) {
  if (err) SLDM_CUDA(cudaMemsetAsync(tp.err.p, 0, sizeof(int), s));
  return err != 0;
}

}  // namespace sldm
