// FP64-accurate block products with several right-hand sides on the tcgen05 tensor
// cores: a complex64 pair of blocks A + Alo (SLDM_PREC_F32X2: 48 bits of the FP64
// operator) times complex128 vectors, for the residuals of iterative refinement and
// sldm_apply.
//
// Error-free slicing (Ozaki, Ogita, Oishi and Rump 2012, in the fixed-point form used on
// matrix units): every 128-column segment of a row of A, and of every column of the
// real-form right-hand side B' (gemm_tc.cu), is scaled by a power of two that takes its
// largest entry into [2^6, 2^7) and cut into seven signed 8-bit digits,
//     a = sum_i a_i 2^-8i,  i = 0 .. 6,  |a_i| <= 128 (an integer; the fourth and fifth, which the
//     pair's second number joins, at most 192).
// Such integers are exact in FP16, their products in FP32, and the sums over 128 columns of the digit
// products of one weight stay within 2^24 for the weights 0 .. 5 (i + j): the tensor core's FP32
// accumulators hold exact integers.  Weight 6 can reach 1.2 x 2^24 if every digit is at its bound; an
// addition beyond 2^24 loses at most a unit of 2^-48, together below 2^-54 of the largest entries' product
// (tests/test_x2_bounds.py).  The products with i + j <= 6
// are kept (28 of 49), level l = i + j in an accumulator of its own; what is left out and
// the digits' tails are below 2^-50 of the segments' largest entries' product, term by term.  The levels of a
// segment are scaled back and added into a compensated pair of FP32 sums (TwoSum for the
// levels 0-3, which carry bits above the pair's first number's last place).  Six digits
// are not enough: rows whose entries lie mostly 10^-2 below their segment's largest lost 2^-42.
//
// On the CUDA cores the same product takes ~44 FP32 operations per complex entry and right-hand
// side (10.9 ms for 13 columns of a 6 x 6 metasurface, N = 34,524); here the entries are cut once
// per pass of up to 16 right-hand sides, ~20 issue slots each in packed FP32: 1.33 ms,
// half the rate of the two blocks' HBM stream (4.2 GB), bound by the split warps' chain.  Its error against
// FP64 is 1/2 to 1/8 of the CUDA-core product's (5e-15 to 6e-14 against 1.3e-14 to 5e-13 by block row).
//
// Roles per CTA as in gemm_tc.cu (tiles, their assignment and the scale exponents of A are
// that plan's): TMA of A and Alo (stages of 64 columns, two boxes each), TMA of the digits
// of B' (boxes of 64 columns x 224 rows: digit j of right-hand side r's two rows at 32 j + 2 r),
// split warps (16 columns per step: digits as FP16 pairs into TMEM), one MMA thread
// (per step seven products: a_i x [b_0 .. b_(6-i)], N = 32 (7 - i), into columns 32 i .. of
// the accumulator; one set of 7 levels is all that fits TMEM beside four operand buffers, and the
// epilogue's drain costs the MMAs ~10% of a segment), epilogue warps.  Every wait is bounded.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>

#include "gemm_x2.h"
#include "tc_ptx.cuh"

namespace sldm {

namespace {

constexpr int X_D = 7;                        // digits, and levels kept
constexpr int X_N = 2 * X2_NRHS;              // accumulator columns of a level
constexpr int X_KS = 16;                      // K columns of a step (one MMA K)
constexpr int X_BOXK = 32;                    // FP32 columns of an A box: one 128-byte swizzle row
constexpr int X_STK = 64;                     // K columns of a stage and of a B' box
constexpr int X_SEG = 128;                    // K columns of a segment
constexpr int X_R = 2;                        // stages in the ring
constexpr int X_NA = 4;                       // A operand buffers (TMEM)
constexpr int X_NBB = 3;                      // B' buffers
constexpr int X_M = 128;
constexpr int X_THREADS = 608;
constexpr uint32_t X_BOX_BYTES = X_M * 128;
constexpr uint32_t X_STAGE_BYTES = 4 * X_BOX_BYTES;  // A 0, A 1, Alo 0, Alo 1
constexpr int X_BROWS = X_D * X_N;                   // 224
constexpr uint32_t X_BBUF = X_BROWS * 128;
constexpr uint32_t X_ACC = X_D * X_N;                // accumulator columns
constexpr uint32_t X_ABUF = X_D * (X_KS / 2);        // operand columns of a step
constexpr uint32_t X_AOP = X_ACC;
static_assert(X_AOP + X_NA * X_ABUF <= 512, "accumulator and operand buffers exceed TMEM");
constexpr int X_NBARS = 2 * X_R + 2 * X_NA + 2 + 2 * X_NBB;
constexpr size_t X_SMEM = size_t(X_R) * X_STAGE_BYTES + size_t(X_NBB) * X_BBUF + 1024 + 512;
static_assert(X_SMEM <= 227 * 1024 && 8 * X_NBARS + 4 <= 512 && X_BBUF % 1024 == 0, "shared memory of a CTA");

__host__ __device__ constexpr uint32_t x_idesc(int n) {  // kind::f16, D FP32, A and B FP16, K-major
  return (1u << 4) | (uint32_t(n >> 3) << 17) | (uint32_t(X_M >> 4) << 24);
}

// the seven digits of (hi + lo) sc of two entries, sc24 = 2^24 sc: rounding to the nearest
// integer by adding and subtracting 1.5 2^23, remainders exact; the low part's integer joins
// the fourth digit and its fraction the remainder, so the fourth and fifth may reach 192
__device__ __forceinline__ void digits(float h0, float h1, float l0, float l1, float sc, float sc24, f2 (&d)[X_D]) {
  const f2 MG = f2_pack(12582912.f, 12582912.f), NM = f2_pack(-12582912.f, -12582912.f), K = f2_pack(256.f, 256.f);
  f2 t = f2_mul(f2_pack(h0, h1), f2_pack(sc, sc));
#pragma unroll
  for (int i = 0; i < X_D; ++i) {
    d[i] = f2_add(f2_add(t, MG), NM);
    if (i < X_D - 1) t = f2_sub(t, d[i]);
    if (i == 3) {
      const f2 l = f2_mul(f2_pack(l0, l1), f2_pack(sc24, sc24)), p = f2_add(f2_add(l, MG), NM);
      d[i] = f2_add(d[i], p);
      t = f2_add(t, f2_sub(l, p));
    }
    if (i < X_D - 1) t = f2_mul(t, K);
  }
}
__device__ __forceinline__ uint32_t pair(f2 v) {
  float a, b;
  f2_unpack(v, a, b);
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ uint32_t pair(float a, float b) {
  const __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&v)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3])
               : "memory");
}
// 4 consecutive columns of this warp's 32 TMEM lanes at each of the seven levels
__device__ __forceinline__ void tmem_ld_levels(uint32_t taddr, f2 (&v)[X_D][2]) {
  uint32_t r[28];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%28];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%4, %5, %6, %7}, [%29];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%8, %9, %10, %11}, [%30];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%12, %13, %14, %15}, [%31];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%16, %17, %18, %19}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%20, %21, %22, %23}, [%33];\n"
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%24, %25, %26, %27}, [%34];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27])
      : "r"(taddr), "r"(taddr + X_N), "r"(taddr + 2 * X_N), "r"(taddr + 3 * X_N), "r"(taddr + 4 * X_N), "r"(taddr + 5 * X_N), "r"(taddr + 6 * X_N)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int l = 0; l < X_D; ++l)
#pragma unroll
    for (int i = 0; i < 2; ++i) v[l][i] = f2_pack(__uint_as_float(r[4 * l + 2 * i]), __uint_as_float(r[4 * l + 2 * i + 1]));
}
__device__ __forceinline__ void two_sum_into(f2& s, f2& c, f2 p) {
  const f2 t = f2_add(s, p), bp = f2_sub(t, s);
  c = f2_add(c, f2_add(f2_sub(s, f2_sub(t, bp)), f2_sub(p, bp)));
  s = t;
}

}  // namespace

// y columns col0 .. col0 + nrhs - 1 (nrhs <= 16) of every job.  aexp: gemm_tc.cu's exponents,
// which aim at [2^14, 2^15): 8 less here.
__global__ void __maxnreg__(96)
    gemm_x2_kernel(const GemvJob* __restrict__ jobs, const unsigned char* __restrict__ maps, const unsigned char* __restrict__ lomaps,
                   const TcTile* __restrict__ tiles, const int32_t* __restrict__ cta_begin, const unsigned char* __restrict__ bmap,
                   const TcJob* __restrict__ tj, const signed char* __restrict__ aexp, const float* __restrict__ bscale,
                   int nrhs, int col0, int* err) {
  extern __shared__ unsigned char x2_raw[];
  const int t_begin = cta_begin[blockIdx.x], t_end = cta_begin[blockIdx.x + 1];
  if (t_begin >= t_end) return;
  const uint32_t raw = smem_u32(x2_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gb = x2_raw + (base - raw);
  const uint32_t bbuf0 = base + X_R * X_STAGE_BYTES;
  const uint32_t bars = bbuf0 + X_NBB * X_BBUF;
  auto full = [&](int s) { return bars + 8u * uint32_t(s); };
  auto empty = [&](int s) { return bars + 8u * uint32_t(X_R + s); };
  auto ready = [&](int b) { return bars + 8u * uint32_t(2 * X_R + b); };
  auto wfree = [&](int b) { return bars + 8u * uint32_t(2 * X_R + X_NA + b); };
  const uint32_t accfull = bars + 8u * uint32_t(2 * X_R + 2 * X_NA), accempty = accfull + 8u;
  auto bfull = [&](int b) { return accempty + 8u * uint32_t(1 + b); };
  auto bfree = [&](int b) { return accempty + 8u * uint32_t(1 + X_NBB + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gb + (bars - base) + 8 * X_NBARS);
  __shared__ int s_fail;
  volatile int* vfail = &s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int q = 0; q < X_R; ++q) {
      mbar_init(full(q), 1);
      mbar_init(empty(q), 8);
    }
    for (int b = 0; b < X_NA; ++b) {
      mbar_init(ready(b), 4);
      mbar_init(wfree(b), 1);
    }
    mbar_init(accfull, 1);
    mbar_init(accempty, 8);
    for (int b = 0; b < X_NBB; ++b) {
      mbar_init(bfull(b), 1);
      mbar_init(bfree(b), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_fail = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // tiles count 32-column sub-chunks in whole segments (4)
  int total = 0;
  for (int t = t_begin; t < t_end; ++t) total += tiles[t].nk;
  const int nstages = total / 2, nsteps = total * 2;

  if (warp == 0) {
    // ---------------- TMA producer of A and Alo
    if (lane == 0) {
      int tile = t_begin, k = 0, nk = tiles[t_begin].nk, st = 0;
      for (; st < nstages; ++st) {
        const int q = st % X_R;
        if (st >= X_R && !mbar_wait(empty(q), uint32_t(((st / X_R) - 1) & 1), vfail)) {
          *vfail = 1;
          break;
        }
        const TcTile T = tiles[tile];
        mbar_expect_tx(full(q), X_STAGE_BYTES);
#pragma unroll
        for (int bx = 0; bx < 4; ++bx)
          tma_load_2d(base + uint32_t(q) * X_STAGE_BYTES + uint32_t(bx) * X_BOX_BYTES,
                      (bx < 2 ? maps : lomaps) + size_t(T.job) * 128, (T.k0 + k + (bx & 1)) * X_BOXK, T.row0, full(q));
        if ((k += 2) == nk) {
          k = 0;
          if (++tile < t_end) nk = tiles[tile].nk;
        }
      }
      for (int q = (st > X_R ? st - X_R : 0); q < st; ++q) mbar_wait(full(q % X_R), uint32_t((q / X_R) & 1));
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer
    if (lane == 0) {
      int last = -1;
      for (int g = 0; g < nsteps; ++g) {
        const int b = g % X_NA, gbx = g / 4, bb = gbx % X_NBB, seg = g / 8, j = g % 8;
        bool ok = true;
        if (j == 0 && seg >= 1) ok = mbar_wait(accempty, uint32_t((seg - 1) & 1), vfail);
        if (ok && (g & 3) == 0) ok = mbar_wait(bfull(bb), uint32_t((gbx / X_NBB) & 1), vfail);
        if (ok) ok = mbar_wait(ready(b), uint32_t((g / X_NA) & 1), vfail);
        if (!ok) {
          *vfail = 1;
          break;
        }
        tc_fence_after();
        const uint32_t aop = tmem + X_AOP + uint32_t(b) * X_ABUF;
        const uint64_t bd = sw128_desc(bbuf0 + uint32_t(bb) * X_BBUF + uint32_t(g & 3) * 32u);
#pragma unroll
        for (int i = 0; i < X_D; ++i)  // digit i of A with digits 0 .. 6 - i of B' into levels i .. 6
          tc_mma_f16(tmem + uint32_t(i * X_N), aop + uint32_t(i * (X_KS / 2)), bd, x_idesc((X_D - i) * X_N),
                     (j > 0 || i > 0) ? 1u : 0u);
        tc_commit(wfree(b));
        if ((g & 3) == 3) tc_commit(bfree(bb));
        if (j == 7) tc_commit(accfull);
        last = g;
      }
      if (last >= 0) {
        mbar_wait(wfree(last % X_NA), uint32_t((last / X_NA) & 1));
        if ((last & 3) == 3) mbar_wait(bfree(last / 4 % X_NBB), uint32_t((last / 4 / X_NBB) & 1));
        if ((last & 7) == 7) mbar_wait(accfull, uint32_t((last / 8) & 1));
      }
    }
    __syncwarp();
  } else if (warp < 10) {
    // ---------------- split warps: thread = row; the two warps of a lane quarter take the steps in turn
    const int q4 = warp & 3, kh = (warp - 2) >> 2, row = 32 * q4 + lane;
    // scale exponents of this row, one segment ahead of their use
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
        ea = aexp + J.aexp + int64_t(T.k0 / 4) * mpad + T.row0 + row;
      }
      const int e = *ea;
      ea += mpad;
      k += 4;
      return e;
    };
    int enext = next_exp();
    float sc = 1.f, sc24 = 1.f;
    for (int g = kh; g < nsteps; g += 2) {
      const int st = g / 4, q = st % X_R, b = g % X_NA;
      if ((g & 7) == kh) {  // this row's scale for the segment
        sc = pow2f(enext - 8);
        sc24 = pow2f(enext + 16);
        enext = next_exp();
      }
      bool ok = mbar_wait(full(q), uint32_t((st / X_R) & 1), vfail);
      if (ok && g >= X_NA) ok = mbar_wait(wfree(b), uint32_t(((g / X_NA) - 1) & 1), vfail);
      ok = __all_sync(0xffffffffu, ok);  // the TMEM stores below need the whole warp
      if (!ok) {
        *vfail = 1;
        break;
      }
      // columns 16 (g % 4) .. + 15 of the stage: box (g % 4) / 2, 16-byte pieces 4 (g % 2) .. + 3
      const unsigned char* rp = gb + size_t(q) * X_STAGE_BYTES + size_t((g & 3) >> 1) * X_BOX_BYTES + size_t(row) * 128;
      const uint32_t ta = tmem + (uint32_t(32 * q4) << 16) + X_AOP + uint32_t(b) * X_ABUF;
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t w[X_D][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int o = ((4 * (g & 1) + 2 * hf + h) ^ (row & 7)) * 16;
          const float4 a = *reinterpret_cast<const float4*>(rp + o);
          const float4 l = *reinterpret_cast<const float4*>(rp + 2 * X_BOX_BYTES + o);
          f2 d0[X_D], d1[X_D];
          digits(a.x, a.y, l.x, l.y, sc, sc24, d0);
          digits(a.z, a.w, l.z, l.w, sc, sc24, d1);
#pragma unroll
          for (int i = 0; i < X_D; ++i) {
            w[i][2 * h] = pair(d0[i]);
            w[i][2 * h + 1] = pair(d1[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < X_D; ++i) tmem_st4(ta + uint32_t(i * (X_KS / 2) + 4 * hf), w[i]);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if ((g & 3) >= 2) mbar_arrive(empty(q));  // this warp's last step of the stage
        mbar_arrive(ready(b));
      }
    }
  } else if (warp == 18) {
    // ---------------- TMA producer of the digits of B'
    if (lane == 0) {
      int tile = t_begin, k = 0, nk = tiles[t_begin].nk, g = 0;
      for (; g < nstages; ++g) {
        const int b = g % X_NBB;
        if (g >= X_NBB && !mbar_wait(bfree(b), uint32_t(((g / X_NBB) - 1) & 1), vfail)) {
          *vfail = 1;
          break;
        }
        mbar_expect_tx(bfull(b), X_BBUF);
        tma_load_2d(bbuf0 + uint32_t(b) * X_BBUF, bmap, 0, X_BROWS * (tj[tiles[tile].job].base + (tiles[tile].k0 + k) / 2), bfull(b));
        if ((k += 2) == nk) {
          k = 0;
          if (++tile < t_end) nk = tiles[tile].nk;
        }
      }
      for (int q = (g > X_NBB ? g - X_NBB : 0); q < g; ++q) mbar_wait(bfull(q % X_NBB), uint32_t((q / X_NBB) & 1));
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps: thread = row, 16 of a level's 32 columns (8 right-hand sides)
    const int q4 = warp & 3, half = (warp - 10) >> 2;
    f2 cs[8], cc[8];  // (re, im) of each
#pragma unroll
    for (int i = 0; i < 8; ++i) cs[i] = cc[i] = 0ull;
    int seg = 0;
    for (int t = t_begin; t < t_end; ++t) {
      const int nseg = tiles[t].nk / 4;
      bool ok = true;
      const signed char* ea;
      const float* eb;
      int mpad;
      {
        const TcTile T = tiles[t];
        const TcJob TJ = tj[T.job];
        mpad = TJ.mpad;
        ea = aexp + TJ.aexp + int64_t(T.k0 / 4) * mpad + T.row0 + 32 * q4 + lane;
        eb = bscale + int64_t(TJ.base / 2 + T.k0 / 4) * X2_NRHS + half * 8 + (lane & 7);
      }
      for (int sg = 0; sg < nseg; ++sg, ++seg) {
        const float sa = pow2f(8 - *ea), sbl = __ldg(eb);  // before the wait for the segment
        ea += mpad;
        eb += X2_NRHS;
        ok = __all_sync(0xffffffffu, mbar_wait(accfull, uint32_t(seg & 1), vfail));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int hq = 0; hq < 4; ++hq) {
          f2 v[X_D][2];
          tmem_ld_levels(tmem + (uint32_t(32 * q4) << 16) + uint32_t(half * 16 + 4 * hq), v);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int c = 2 * hq + i;
            const float sb = __shfl_sync(0xffffffffu, sbl, c);
            const f2 a2 = f2_pack(sa, sa);
            auto k = [&](float w) { return f2_pack(sb * w, sb * w); };
            two_sum_into(cs[c], cc[c], f2_mul(f2_mul(v[0][i], a2), k(1.f)));
            two_sum_into(cs[c], cc[c], f2_mul(f2_mul(v[1][i], a2), k(0x1p-8f)));
            two_sum_into(cs[c], cc[c], f2_mul(f2_mul(v[2][i], a2), k(0x1p-16f)));
            two_sum_into(cs[c], cc[c], f2_mul(f2_mul(v[3][i], a2), k(0x1p-24f)));
            // levels 4-6 lie below the first sum's last place
            const f2 h = f2_pack(0x1p-8f, 0x1p-8f);
            cc[c] = f2_fma(f2_mul(f2_fma(f2_fma(v[6][i], h, v[5][i]), h, v[4][i]), a2), k(0x1p-32f), cc[c]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(accempty);
      }
      if (!ok) {
        *vfail = 1;
        break;
      }
      const TcTile T = tiles[t];
      const GemvJob& J = jobs[T.job];
      const int row = T.row0 + 32 * q4 + lane;
      if (row < J.m) {
        double2* y = reinterpret_cast<double2*>(J.y) + int64_t(col0) * J.ldy + row;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const int r = half * 8 + c;
          if (r < nrhs) {
            float s0, s1, c0, c1;
            f2_unpack(cs[c], s0, s1);
            f2_unpack(cc[c], c0, c1);
            const double re = double(s0) + double(c0), im = double(s1) + double(c1);
            double2 o = make_double2(J.ar * re - J.ai * im, J.ar * im + J.ai * re);
            double2* yy = y + int64_t(r) * J.ldy;
            if (T.split) {  // one of the two K halves of the tile (Y zeroed before the pass)
              atomicAdd(&yy->x, o.x);
              atomicAdd(&yy->y, o.y);
            } else {
              if (J.beta) {
                const double2 p = *yy;
                o.x += p.x;
                o.y += p.y;
              }
              *yy = o;
            }
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) cs[i] = cc[i] = 0ull;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0 && *vfail) atomicExch(err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// Digits of B' of one segment (64 complex columns, two boxes) per block: 8 threads per
// right-hand side, 8 columns each; x as a float pair hi + lo (48 bits).  bscale[segment][r] undoes
// the scale.  Blocks nstage and above zero the Y rows of the tiles split along K.
__global__ void __launch_bounds__(128) x2_bprime_kernel(const GemvJob* __restrict__ jobs, const int32_t* __restrict__ gjob,
                                                        const int32_t* __restrict__ gst, int nstage,
                                                        const TcTile* __restrict__ ztiles, int nrhs, int col0,
                                                        __half* __restrict__ bp, float* __restrict__ bscale) {
  const int gidx = blockIdx.x;
  if (gidx >= nstage) {
    const TcTile T = ztiles[gidx - nstage];
    const GemvJob& J = jobs[T.job];
    double2* y = reinterpret_cast<double2*>(J.y) + int64_t(col0) * J.ldy;
    for (int e = threadIdx.x; e < X_M * nrhs; e += blockDim.x) {
      const int row = T.row0 + e % X_M, r = e / X_M;
      if (row < J.m) y[int64_t(r) * J.ldy + row] = make_double2(0.0, 0.0);
    }
    return;
  }
  const GemvJob& J = jobs[gjob[gidx]];
  const int r = threadIdx.x >> 3, sub = threadIdx.x & 7, c0 = gst[gidx] * (X_SEG / 2) + sub * 8;
  const double2* x = reinterpret_cast<const double2*>(J.x) + int64_t(col0 + r) * J.ldx;
  float2 h[8], l[8];
  float m = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const double2 v = r < nrhs && c0 + i < J.n ? x[c0 + i] : make_double2(0.0, 0.0);
    h[i] = make_float2(__double2float_rn(v.x), __double2float_rn(v.y));
    l[i] = make_float2(__double2float_rn(v.x - double(h[i].x)), __double2float_rn(v.y - double(h[i].y)));
    m = fmaxf(m, fmaxf(fabsf(h[i].x), fabsf(h[i].y)));
  }
  for (int o = 4; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = tc_scale_exp(m) - 8;
  const float sc = pow2f(e), sc24 = pow2f(e + 24);
  if (sub == 0) bscale[int64_t(gidx) * X2_NRHS + r] = pow2f(-e);
  uint32_t w0[X_D][8], w1[X_D][8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    f2 d[X_D];
    digits(h[i].x, h[i].y, l[i].x, l[i].y, sc, sc24, d);
#pragma unroll
    for (int j = 0; j < X_D; ++j) {
      float re, im;
      f2_unpack(d[j], re, im);
      w0[j][i] = pair(f2_pack(re, -im));
      w1[j][i] = pair(f2_pack(im, re));
    }
  }
  __half* box = bp + (size_t(2 * gidx + (sub >> 2)) * X_BROWS) * X_STK + 16 * (sub & 3);
#pragma unroll
  for (int j = 0; j < X_D; ++j) {
    uint4* p0 = reinterpret_cast<uint4*>(box + size_t(j * X_N + 2 * r) * X_STK);
    uint4* p1 = reinterpret_cast<uint4*>(box + size_t(j * X_N + 2 * r + 1) * X_STK);
    p0[0] = make_uint4(w0[j][0], w0[j][1], w0[j][2], w0[j][3]);
    p0[1] = make_uint4(w0[j][4], w0[j][5], w0[j][6], w0[j][7]);
    p1[0] = make_uint4(w1[j][0], w1[j][1], w1[j][2], w1[j][3]);
    p1[1] = make_uint4(w1[j][4], w1[j][5], w1[j][6], w1[j][7]);
  }
}

// ---------------------------------------------------------------- host side
void x2_plan_build(const std::vector<GemvJob>& jobs, const TcPlan& tc, X2Plan& xp, cudaStream_t s) {
  xp.ok = false;
  if (!tc.ok || jobs.empty()) return;
  // A pass takes ~6.6 us per segment of the fullest CTA (and the launches ~12 us) whatever
  // its width up to 16, the CUDA cores ~3 ps per entry and right-hand side.  Whole products, tensor against
  // CUDA cores: 6 x 6 metasurface, 3 right-hand sides 1,383 / 1,958 us, 16: 1,437 / 10,803; 3 x 3, 3:
  // 229 / 224, 4: 229 / 275; a sphere of 320 triangles, 8: 120 / 95, 16: 126 / 130.
  double entries = 0;
  for (const auto& J : jobs) entries += double(J.m) * J.n;
  const int forced = tc_policy();
  xp.from = forced ? forced : std::max(2, int(std::ceil((12.0 + 6.6 * tc.longest) / (3e-6 * entries))));
  if (xp.from > X2_NRHS) return;
  std::vector<unsigned char> maps(jobs.size() * 128);
  for (size_t i = 0; i < jobs.size(); ++i) {
    const GemvJob& J = jobs[i];
    if (J.Alo == nullptr || !tc_block_map(J.Alo, J.lda, J.m, J.n, &maps[i * 128])) return;
  }
  xp.bprime.alloc(size_t(tc.nstage) * 2 * X_BROWS * X_STK);
  xp.bscale.alloc(size_t(tc.nstage) * X2_NRHS);
  std::vector<unsigned char> bm(128);
  if (!tc_map_2d(CU_TENSOR_MAP_DATA_TYPE_FLOAT16, xp.bprime.p, X_STK, uint64_t(tc.nstage) * 2 * X_BROWS, X_STK * 2, X_STK, X_BROWS,
                 bm.data()))
    return;
  xp.lomaps.upload(maps, s);
  xp.bmap.upload(bm, s);
  xp.tc = &tc;
  SLDM_CUDA(cudaStreamSynchronize(s));
  xp.ok = true;
}

void gemm_x2(const GemvPlan& plan, const X2Plan& xp, int nrhs, int col0, cudaStream_t s) {
  SLDM_REQUIRE(xp.ok && nrhs >= 1 && nrhs <= X2_NRHS, SLDM_EINVAL, "FP64-accurate tensor-core product: invalid plan or nrhs");
  static std::atomic<uint64_t> attr_set{0};
  int dev = 0;
  SLDM_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (!(attr_set.load() & bit)) {
    SLDM_CUDA(cudaFuncSetAttribute(gemm_x2_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(X_SMEM)));
    attr_set.fetch_or(bit);
  }
  const TcPlan& tc = *xp.tc;
  x2_bprime_kernel<<<unsigned(tc.nstage + tc.nzero), 128, 0, s>>>(plan.jobs, tc.gjob.p, tc.gst.p, tc.nstage, tc.ztiles.p, nrhs, col0,
                                                                  reinterpret_cast<__half*>(xp.bprime.p), xp.bscale.p),
      count_launch();
  gemm_x2_kernel<<<unsigned(tc.nctas), X_THREADS, X_SMEM, s>>>(plan.jobs, tc.maps.p, xp.lomaps.p, tc.tiles.p, tc.cta_begin.p,
                                                               xp.bmap.p, tc.tj.p, tc.aexp.p, xp.bscale.p, nrhs, col0, tc.err.p),
      count_launch();
  SLDM_CUDA(cudaGetLastError());
  tc.ran = true;
  if (take_tc_wait()) SLDM_CUDA(cudaMemsetAsync(tc.err.p, 1, sizeof(int), s));
}

}  // namespace sldm
