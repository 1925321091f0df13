// Blocked right-looking LU with partial pivoting: A X = B in place, A n x n and B
// n x r, row-major.  Per panel of NB columns:
//
//   1. lu_panel_cluster  factor the panel [j0, j0 + nb) over rows j0..n-1: one cluster of
//                        CTAs, each with a contiguous chunk of the panel's rows in
//                        shared memory; per column one cluster barrier, after
//                        which every CTA reads the candidates' pivots and the pivot
//                        row through distributed shared memory.  (Panels taller than
//                        the cluster's shared memory: lu_panel_kernel, a cooperative
//                        launch with two bounded grid barriers per column.)
//   2. lu_solve_kernel   on the columns right of the panel and on B: the panel's row
//                        interchanges (as one gather) and X = L11^-1 X (unit lower);
//                        the L columns left of the panel are never read again;
//   3. lu_gemm           A22 -= L21 U12 on the trailing rows of those columns.
//
// then back substitution U X = B panel by panel from the bottom (upper triangular
// solve on the panel's rows, GEMM update of the rows above).
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "cluster.h"
#include "dense.h"
#include "widen.cuh"

namespace sldm {

namespace {

// Panel width: the panel costs ~2 us a column whatever its width, the FP64 kernels work
// on half the columns at a time for shared memory
template <class C>
constexpr int panel_width() {
  return sizeof(C) == 8 ? 64 : 32;
}
constexpr int NB_MAX = 64;
constexpr int PANEL_THREADS = 256;
constexpr int PANEL_MIN_ROWS = 32;   // rows per CTA of the panel factorisation, at least
constexpr unsigned SPIN_LIMIT = 1u << 22;

template <class C>
struct CT2;
template <>
struct CT2<float2> {
  typedef float R;
};
template <>
struct CT2<double2> {
  typedef double R;
};

template <class C>
__device__ __forceinline__ C cmul_(C a, C b) {
  C r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
template <class C>
__device__ __forceinline__ C cdiv_(C a, C b) {
  typedef typename CT2<C>::R R;
  const R d = b.x * b.x + b.y * b.y;
  C r;
  r.x = (a.x * b.x + a.y * b.y) / d;
  r.y = (a.y * b.x - a.x * b.y) / d;
  return r;
}

// acc += a b and acc -= a b for complex numbers as chains of fused multiply-adds
template <class R>
__device__ __forceinline__ void cfma(R& cr, R& ci, R ar, R ai, R br, R bi) {
  cr = fma(ar, br, cr);
  cr = fma(-ai, bi, cr);
  ci = fma(ar, bi, ci);
  ci = fma(ai, br, ci);
}
template <class R>
__device__ __forceinline__ void cfms(R& cr, R& ci, R ar, R ai, R br, R bi) {
  cr = fma(-ar, br, cr);
  cr = fma(ai, bi, cr);
  ci = fma(-ar, bi, ci);
  ci = fma(-ai, br, ci);
}

__device__ __forceinline__ unsigned ld_acq(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid barrier over the launch's CTAs (all co-resident: cooperative launch).
// Bounded: a wait that runs out sets *err = 2; every CTA then leaves at its next
// barrier.  Returns false when the kernel must stop (CTA-uniform).
__device__ bool grid_barrier(unsigned* ctr, unsigned target, int* err) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(ctr, 1u);
    int ok = 1;
    unsigned it = 0;
    while (ld_acq(ctr) < target) {
      if (*(volatile int*)err) { ok = 0; break; }
      if (++it > SPIN_LIMIT) { atomicExch(err, 2); ok = 0; break; }
      __nanosleep(32);
    }
    s_ok = ok && !*(volatile int*)err;
  }
  __syncthreads();
  return s_ok != 0;
}

// Injected failure (sldm_test_inject): a bounded wait for a flag that nothing sets, on the solver's own error
// record; every kernel after it leaves at once, as after a panel's barrier that ran out.
__global__ void lu_stall_kernel(const unsigned* flag, int* err) {
  for (unsigned it = 0; it < SPIN_LIMIT / 8; ++it) {
    if (ld_acq(flag)) return;
    __nanosleep(32);
  }
  atomicExch(err, 2);
}

// ---------------------------------------------------------------- 1. panel
// CTA c holds rows [j0 + c*chunk, min(n, j0 + (c+1)*chunk)) of columns
// [j0, j0 + nb) in shared memory.  Pivot candidates go to slot_v/slot_i[c];
// the pivot row and the current row travel through urow/orow.
template <class C>
__global__ void __launch_bounds__(PANEL_THREADS) lu_panel_kernel(C* A, int n, int j0, int nb, int chunk, int* piv,
                                                                 C* urow, C* orow, double* slot_v, int* slot_i,
                                                                 unsigned* bar, int* err) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);  // chunk x nb
  C* U = P + size_t(chunk) * nb;          // nb: the current U row
  __shared__ double s_bv[PANEL_THREADS / 32];
  __shared__ int s_bi[PANEL_THREADS / 32];
  __shared__ int s_p;
  const int G = gridDim.x, c = blockIdx.x;
  if (*(volatile int*)err) return;  // an earlier panel failed (uniform across the grid)
  const int r0 = j0 + c * chunk, r1 = min(n, r0 + chunk), nr = max(0, r1 - r0);
  for (int t = threadIdx.x; t < nr * nb; t += blockDim.x) {
    const int i = t / nb, j = t % nb;
    P[t] = A[int64_t(r0 + i) * n + j0 + j];
  }
  __syncthreads();  // the pivot search reads rows loaded by other threads
  unsigned epoch = 0;
  for (int j = 0; j < nb; ++j) {
    const int J = j0 + j;
    // local pivot candidate over rows >= J: largest |a|^2, smallest row on ties
    double best = -1.0;
    int bi = n;
    for (int i = threadIdx.x; i < nr; i += blockDim.x) {
      const int row = r0 + i;
      if (row < J) continue;
      const C a = P[size_t(i) * nb + j];
      const double v = double(a.x) * double(a.x) + double(a.y) * double(a.y);
      if (v > best || (v == best && row < bi)) { best = v; bi = row; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if ((threadIdx.x & 31) == 0) { s_bv[threadIdx.x >> 5] = best; s_bi[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < int(blockDim.x >> 5); ++w)
        if (s_bv[w] > s_bv[0] || (s_bv[w] == s_bv[0] && s_bi[w] < s_bi[0])) { s_bv[0] = s_bv[w]; s_bi[0] = s_bi[w]; }
      slot_v[c] = s_bv[0];
      slot_i[c] = s_bi[0];
    }
    if (!grid_barrier(bar, (++epoch) * G, err)) return;
    if (threadIdx.x < 32) {  // warp 0 reduces the G candidates (loads in parallel)
      double b = -1.0;
      int p = n;
      for (int g = threadIdx.x; g < G; g += 32) {
        const double v = __ldcg(slot_v + g);
        const int i = __ldcg(slot_i + g);
        if (v > b || (v == b && i < p)) { b = v; p = i; }
      }
      for (int o = 16; o > 0; o >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, b, o);
        const int oi = __shfl_xor_sync(0xffffffffu, p, o);
        if (ob > b || (ob == b && oi < p)) { b = ob; p = oi; }
      }
      if (threadIdx.x == 0) {
        s_p = (b > 0.0 && p < n) ? p : -1;  // zero, non-finite or missing pivot
        if (s_p < 0 && c == 0) {
          err[1] = J;  // where it stopped
          atomicExch(err, 1);
        }
        if (c == 0 && s_p >= 0) piv[J] = s_p;
      }
    }
    __syncthreads();
    const int p = s_p;
    if (p < 0) return;  // CTA-uniform; the others stop at their next barrier
    // the owners publish the pivot row and the current row
    if (p >= r0 && p < r1)
      for (int t = threadIdx.x; t < nb; t += blockDim.x) urow[t] = P[size_t(p - r0) * nb + t];
    if (J >= r0 && J < r1)
      for (int t = threadIdx.x; t < nb; t += blockDim.x) orow[t] = P[size_t(J - r0) * nb + t];
    if (!grid_barrier(bar, (++epoch) * G, err)) return;
    for (int t = threadIdx.x; t < nb; t += blockDim.x) U[t] = __ldcg(urow + t);
    __syncthreads();
    if (p != J && p >= r0 && p < r1)
      for (int t = threadIdx.x; t < nb; t += blockDim.x) P[size_t(p - r0) * nb + t] = __ldcg(orow + t);
    if (J >= r0 && J < r1)
      for (int t = threadIdx.x; t < nb; t += blockDim.x) P[size_t(J - r0) * nb + t] = U[t];
    __syncthreads();
    // multipliers of the rows below J, then the rank-1 update of the panel's remaining columns
    const C piv_v = U[j];
    for (int i = threadIdx.x; i < nr; i += blockDim.x)
      if (r0 + i > J) P[size_t(i) * nb + j] = cdiv_(P[size_t(i) * nb + j], piv_v);
    __syncthreads();
    const int w = nb - j - 1;
    if (w > 0)
      for (int t = threadIdx.x; t < nr * w; t += blockDim.x) {
        const int i = t / w, cc = 1 + t % w;
        if (r0 + i <= J) continue;
        const C l = P[size_t(i) * nb + j], u = U[j + cc];
        C a = P[size_t(i) * nb + j + cc];
        cfms(a.x, a.y, l.x, l.y, u.x, u.y);
        P[size_t(i) * nb + j + cc] = a;
      }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < nr * nb; t += blockDim.x) {
    const int i = t / nb, j = t % nb;
    A[int64_t(r0 + i) * n + j0 + j] = P[t];
  }
}

// ---------------------------------------------------------------- 1. panel, one cluster
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// address, in the shared memory of CTA `rank`, of this CTA's variable at p
__device__ __forceinline__ unsigned in_cta(const void* p, unsigned rank) {
  unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p)), b;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  return b;
}
__device__ __forceinline__ unsigned long long ld_cta_u64(unsigned a) {
  unsigned long long v;
  asm volatile("ld.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void ld_cta(unsigned a, float2& v) {
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
}
__device__ __forceinline__ void ld_cta(unsigned a, double2& v) {
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a));
}

// Row moves of a panel: row j0 + j receives row in[j]; row out_row[k] (below the panel's
// block, -1: none) receives row out_src[k].
struct Moves {
  int in[NB_MAX], out_row[NB_MAX], out_src[NB_MAX];
};
// The net effect of swapping row j0 + j with piv[j], j = 0 .. nb - 1, by one warp.
__device__ void net_moves(Moves& m, const int* piv, int j0, int nb) {
  const int lane = threadIdx.x & 31;
  for (int j = lane; j < NB_MAX; j += 32) {
    m.in[j] = j0 + j;
    m.out_row[j] = m.out_src[j] = -1;
  }
  __syncwarp();
  for (int j = 0; j < nb; ++j) {
    const int p = piv[j];
    if (p != j0 + j) {
      int at = -1;  // the entry of an outside row already moved
      for (int b = 0; b < NB_MAX; b += 32) {
        const unsigned hit = __ballot_sync(0xffffffffu, m.out_row[b + lane] == p);
        if (hit) at = b + __ffs(hit) - 1;
      }
      if (lane == 0) {
        const int mine = m.in[j];
        if (p < j0 + nb) {
          m.in[j] = m.in[p - j0];
          m.in[p - j0] = mine;
        } else if (at >= 0) {
          m.in[j] = m.out_src[at];
          m.out_src[at] = mine;
        } else {
          m.out_row[j] = p;
          m.out_src[j] = mine;
          m.in[j] = p;
        }
      }
    }
    __syncwarp();
  }
}
__global__ void lu_moves_kernel(const int* __restrict__ piv, int j0, int nb, Moves* out, const int* __restrict__ err) {
  __shared__ Moves m;
  if (*err) return;
  net_moves(m, piv + j0, j0, nb);
  __syncwarp();
  for (int i = threadIdx.x; i < int(sizeof(Moves) / sizeof(int)); i += 32)
    reinterpret_cast<int*>(out)[i] = reinterpret_cast<const int*>(&m)[i];
}

// A pivot candidate as one integer: |Re| + |Im| (32 leading bits: the choice is within 2^-20
// of the largest) above the complement of the row, so the maximum is the largest value
// and, on ties, the smallest row.  A non-finite value is above every finite one: the
// maximum finds it and pivot_ok refuses it.  0 is no candidate.
__device__ __forceinline__ unsigned long long pivot_key(float2 a, int row) {
  const unsigned v = __float_as_uint(fabsf(a.x) + fabsf(a.y));
  return ((unsigned long long)v << 32) | unsigned(~row);
}
__device__ __forceinline__ unsigned long long pivot_key(double2 a, int row) {
  const unsigned v = unsigned(__double2hiint(fabs(a.x) + fabs(a.y)));
  return ((unsigned long long)v << 32) | unsigned(~row);
}
__device__ __forceinline__ bool pivot_ok(unsigned long long key, float) { return (key >> 32) - 1 < 0x7f800000u - 1; }
__device__ __forceinline__ bool pivot_ok(unsigned long long key, double) { return (key >> 32) - 1 < 0x7ff00000u - 1; }
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}

// CTA of rank c holds rows [j0 + c chunk, ..) in shared memory.  Per column: the largest
// candidate of its rows (integer compares), candidate and rows
// published, one cluster barrier, then every CTA picks the winner, takes the pivot row and
// updates its rows.  Publication buffers alternate: a CTA writes buffer b again only
// after the next column's barrier, which all reach having read b.
// The 50 panels of a complex64 system of n = 3,199: 24.1 ms with two grid barriers through
// global memory -> 10.8 ms in a cluster -> 8.4 ms with integer keys and four barriers of the CTA per column.
constexpr int PC_THREADS = 512;
template <class C, int CS>
__global__ void __launch_bounds__(PC_THREADS) lu_panel_cluster(C* A, int n, int j0, int nb, int chunk, Moves* moves, int* err) {
  typedef typename CT2<C>::R R;
  constexpr int LD = panel_width<C>() + 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* P = reinterpret_cast<C*>(smem_raw);  // chunk x LD
  __shared__ __align__(16) C crow[2][NB_MAX], orow[2][NB_MAX], U[NB_MAX];
  __shared__ unsigned long long cand[2], wv[PC_THREADS / 32];
  __shared__ int s_win, s_p, piv[NB_MAX];
  __shared__ C s_inv;
  __shared__ Moves mv;
  if (*(volatile int*)err) return;  // an earlier panel failed (uniform across the grid)
  const int rank = int(cluster_rank());
  const int r0 = j0 + rank * chunk, nr = max(0, min(n, r0 + chunk) - r0);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int t = threadIdx.x; t < nr * nb; t += PC_THREADS) {
    const int i = t / nb, j = t % nb;
    P[i * LD + j] = A[int64_t(r0 + i) * n + j0 + j];
  }
  __syncthreads();
  bool failed = false;
  for (int j = 0; j < nb; ++j) {
    const int J = j0 + j, buf = j & 1;
    unsigned long long best = 0;
    for (int i = threadIdx.x; i < nr; i += PC_THREADS)
      if (r0 + i >= J) {
        const unsigned long long v = pivot_key(P[i * LD + j], r0 + i);
        best = v > best ? v : best;
      }
    best = warp_max(best);
    if (lane == 0) wv[warp] = best;
    __syncthreads();
    best = warp_max(lane < PC_THREADS / 32 ? wv[lane] : 0);  // every warp for itself
    if (threadIdx.x == 0) cand[buf] = best;
    if (best != 0)
      for (int t = threadIdx.x; t < nb; t += PC_THREADS) crow[buf][t] = P[(int(~unsigned(best)) - r0) * LD + t];
    if (J >= r0 && J < r0 + nr)
      for (int t = threadIdx.x; t < nb; t += PC_THREADS) orow[buf][t] = P[(J - r0) * LD + t];
    cluster_sync();
    if (warp == 0) {
      const unsigned long long mine = lane < CS ? ld_cta_u64(in_cta(&cand[buf], lane)) : 0;
      const unsigned long long v = warp_max(mine);
      const int w = __ffs(__ballot_sync(0xffffffffu, mine == v && lane < CS)) - 1;
      const bool ok = pivot_ok(v, R());
      for (int t = lane; t < nb && ok; t += 32) {  // the pivot row, from its CTA
        C u;
        ld_cta(in_cta(&crow[buf][t], w), u);
        U[t] = u;
      }
      __syncwarp();
      if (lane == 0) {
        s_win = w;
        s_p = ok ? int(~unsigned(v)) : -1;
        if (ok) {
          piv[j] = int(~unsigned(v));
          C one;
          one.x = R(1);
          one.y = R(0);
          s_inv = cdiv_(one, U[j]);
        } else if (rank == 0) {  // zero, non-finite or missing pivot
          err[1] = J;
          atomicExch(err, 1);
        }
      }
    }
    __syncthreads();
    const int p = s_p;
    if (p < 0) {  // the same in every CTA
      failed = true;
      break;
    }
    // rows J and p change places
    if (p != J && rank == s_win)
      for (int t = threadIdx.x; t < nb; t += PC_THREADS) {
        C o;
        ld_cta(in_cta(&orow[buf][t], (J - j0) / chunk), o);
        P[(p - r0) * LD + t] = o;
      }
    if (J >= r0 && J < r0 + nr)
      for (int t = threadIdx.x; t < nb; t += PC_THREADS) P[(J - r0) * LD + t] = U[t];
    __syncthreads();
    // multipliers of the rows below J, then the rank-1 update of the remaining columns
    const C inv = s_inv;
    const int lo = max(0, J + 1 - r0);  // first row below J
    for (int i = lo + threadIdx.x; i < nr; i += PC_THREADS) P[i * LD + j] = cmul_(P[i * LD + j], inv);
    __syncthreads();
    if constexpr (sizeof(C) == 16) {
      // FP64: full warps whatever the column count (an instruction costs 16 clocks however many lanes it serves)
      const int w = nb - j - 1, work = (nr - lo) * w;
      for (int t = threadIdx.x; t < work; t += PC_THREADS) {
        const int i = lo + t / w, cc = j + 1 + t % w;
        const C l = P[i * LD + j], u = U[cc];
        C a = P[i * LD + cc];
        cfms(a.x, a.y, l.x, l.y, u.x, u.y);
        P[i * LD + cc] = a;
      }
    } else for (int c0 = j + 1; c0 < nb; c0 += 32) {  // a warp takes a row, its lanes the columns
      const int cc = c0 + lane;
      if (cc >= nb) continue;
      const C u = U[cc];
#pragma unroll 4
      for (int i = lo + warp; i < nr; i += PC_THREADS / 32) {
        const C l = P[i * LD + j];
        C a = P[i * LD + cc];
        cfms(a.x, a.y, l.x, l.y, u.x, u.y);
        P[i * LD + cc] = a;
      }
    }
    __syncthreads();
  }
  if (!failed) {
    for (int t = threadIdx.x; t < nr * nb; t += PC_THREADS) {
      const int i = t / nb, j = t % nb;
      A[int64_t(r0 + i) * n + j0 + j] = P[i * LD + j];
    }
    if (rank == 0 && warp == 0) {
      net_moves(mv, piv, j0, nb);
      __syncwarp();
      for (int i = lane; i < int(sizeof(Moves) / sizeof(int)); i += 32)
        reinterpret_cast<int*>(moves)[i] = reinterpret_cast<const int*>(&mv)[i];
    }
  }
  cluster_sync();  // no CTA leaves while another may read its shared memory
}

// Columns right of the panel: A's columns [ca, n) then B's columns [0, r).
template <class C>
struct Cols {
  C* A;
  int n, ca;
  C* B;
  int r;
  __device__ __forceinline__ int count() const { return (n - ca) + r; }
  // pointer to row 0 of column q of the set, and its row stride
  __device__ __forceinline__ C* col(int q, int64_t& ld) const {
    if (q < n - ca) {
      ld = n;
      return A + ca + q;
    }
    ld = r;
    return B + (q - (n - ca));
  }
};

// ---------------------------------------------------------------- 2. interchanges and triangular solve
// LOWER: the panel's row moves, then X = L11^-1 X (unit lower); else X = U11^-1 X (upper).
// A CTA takes 32 columns; the triangle and the columns' rows lie in shared memory, and
// column j of the triangle updates the rows not yet final, spread over all threads (one
// thread per column ran a chain of nb^2 / 2 FP64 products on one lane each: 308 us per
// 64-row FP64 panel, and its row swaps 23 us; this takes 28 us per 32 rows, swaps included).
constexpr int TS_COLS = 32, TS_THREADS = 256;
template <class C, bool LOWER>
__global__ void __launch_bounds__(TS_THREADS) lu_solve_kernel(Cols<C> S, const C* __restrict__ A, int n, int j0, int nb,
                                                              const Moves* __restrict__ mv, const int* __restrict__ err) {
  if (*err) return;
  constexpr int NBW = panel_width<C>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* T = reinterpret_cast<C*>(smem_raw);  // nb x (NBW + 1)
  C* X = T + NBW * (NBW + 1);             // nb x TS_COLS
  C* O = X + NBW * TS_COLS;               // LOWER: the rows that go below the block
  __shared__ C inv[NB_MAX];
  const int c = threadIdx.x % TS_COLS, rr = threadIdx.x / TS_COLS;
  constexpr int RG = TS_THREADS / TS_COLS;  // row groups
  const int q = blockIdx.x * TS_COLS + c;
  const bool mine = q < S.count();
  int64_t ld = 0;
  C* col = mine ? S.col(q, ld) : nullptr;
  for (int e = threadIdx.x; e < nb * nb; e += TS_THREADS) T[(e / nb) * (NBW + 1) + e % nb] = A[int64_t(j0 + e / nb) * n + j0 + e % nb];
  for (int k = rr; k < nb; k += RG) {
    if (mine) X[k * TS_COLS + c] = col[int64_t(LOWER ? mv->in[k] : j0 + k) * ld];
    if (LOWER && mine && mv->out_row[k] >= 0) O[k * TS_COLS + c] = col[int64_t(mv->out_src[k]) * ld];
  }
  __syncthreads();
  if (LOWER) {
    for (int k = rr; k < nb; k += RG)
      if (mine && mv->out_row[k] >= 0) col[int64_t(mv->out_row[k]) * ld] = O[k * TS_COLS + c];
    for (int j = 0; j + 1 < nb; ++j) {
      const C x = X[j * TS_COLS + c];
      for (int i = j + 1 + rr; i < nb; i += RG) {
        const C l = T[i * (NBW + 1) + j];
        C v = X[i * TS_COLS + c];
        cfms(v.x, v.y, l.x, l.y, x.x, x.y);
        X[i * TS_COLS + c] = v;
      }
      __syncthreads();
    }
    for (int k = rr; k < nb; k += RG)
      if (mine) col[int64_t(j0 + k) * ld] = X[k * TS_COLS + c];
  } else {
    if (threadIdx.x < nb) {
      C one;
      one.x = 1;
      one.y = 0;
      inv[threadIdx.x] = cdiv_(one, T[threadIdx.x * (NBW + 1) + threadIdx.x]);
    }
    __syncthreads();
    for (int j = nb - 1; j >= 0; --j) {
      const C x = cmul_(X[j * TS_COLS + c], inv[j]);
      if (mine && rr == 0) col[int64_t(j0 + j) * ld] = x;
      for (int i = rr; i < j; i += RG) {
        const C u = T[i * (NBW + 1) + j];
        C v = X[i * TS_COLS + c];
        cfms(v.x, v.y, u.x, u.y, x.x, x.y);
        X[i * TS_COLS + c] = v;
      }
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- 3. trailing update
// X[i, q] -= sum_k P[i, k] Q[k, q] for rows i in [i0, i1) of the column set,
// P[i, k] = A[i, kc + k], Q[k, q] = column q of the set at row k0 + k, k < nb.
// A CTA of 256 threads makes a TM x TN tile, TM / 16 x TN / 16 results per thread (columns
// interleaved).  FP64: bound by the FP64 pipe (64 x 64 tiles, 92% busy); a trailing block of
// few tiles takes 32 x 32 ones to reach every SM.  Complex64: packed FP32 pairs, two
// fma.rn.f32x2 per complex product, two k per step (the scalar form ran at 28 TFLOP/s).
__device__ __forceinline__ unsigned long long pk(float lo, float hi) {
  unsigned long long u;
  asm("mov.b64 %0, {%1, %2};" : "=l"(u) : "f"(lo), "f"(hi));
  return u;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
template <class C, int TM, int TN>
__global__ void __launch_bounds__(256) lu_gemm_kernel(Cols<C> S, const C* __restrict__ A, int n, int i0, int i1, int kc,
                                                      int k0, int nb, const int* __restrict__ err) {
  if (*err) return;
  constexpr int NBW = panel_width<C>(), LDP = NBW + 16 / int(sizeof(C));  // 16-byte aligned rows, shifted banks
  constexpr int RM = TM / 16, RN = TN / 16;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* Ps = reinterpret_cast<C*>(smem_raw);  // TM x LDP
  C* Qs = Ps + TM * LDP;                   // NBW x TN
  const int rt = i0 + blockIdx.y * TM, qt = blockIdx.x * TN;
  const int nq = S.count();
  C zero;
  zero.x = 0;
  zero.y = 0;
  for (int t = threadIdx.x; t < TM * NBW; t += 256) {
    const int i = t / NBW, k = t % NBW;
    Ps[i * LDP + k] = rt + i < i1 && k < nb ? A[int64_t(rt + i) * n + kc + k] : zero;
  }
  for (int t = threadIdx.x; t < NBW * TN; t += 256) {
    const int k = t / TN, q = t % TN;
    C v = zero;
    if (qt + q < nq && k < nb) {
      int64_t ld;
      const C* col = S.col(qt + q, ld);
      v = col[int64_t(k0 + k) * ld];
    }
    Qs[t] = v;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if constexpr (sizeof(C) == 8) {
    unsigned long long acc[RM][RN];
#pragma unroll
    for (int a = 0; a < RM; ++a)
#pragma unroll
      for (int b = 0; b < RN; ++b) acc[a][b] = 0ull;
    for (int k = 0; k < nb; k += 2) {  // rows and columns from nb on are zero
      float4 p[RM];
      float2 q0[RN], q1[RN];
#pragma unroll
      for (int a = 0; a < RM; ++a) p[a] = *reinterpret_cast<const float4*>(&Ps[(ty * RM + a) * LDP + k]);
#pragma unroll
      for (int b = 0; b < RN; ++b) {
        q0[b] = Qs[k * TN + tx + 16 * b];
        q1[b] = Qs[(k + 1) * TN + tx + 16 * b];
      }
#pragma unroll
      for (int b = 0; b < RN; ++b) {
        const unsigned long long x0 = pk(q0[b].x, q0[b].y), y0 = pk(-q0[b].y, q0[b].x);
        const unsigned long long x1 = pk(q1[b].x, q1[b].y), y1 = pk(-q1[b].y, q1[b].x);
#pragma unroll
        for (int a = 0; a < RM; ++a) {
          fma2(acc[a][b], pk(p[a].x, p[a].x), x0);
          fma2(acc[a][b], pk(p[a].y, p[a].y), y0);
          fma2(acc[a][b], pk(p[a].z, p[a].z), x1);
          fma2(acc[a][b], pk(p[a].w, p[a].w), y1);
        }
      }
    }
#pragma unroll
    for (int b = 0; b < RN; ++b) {
      const int qq = qt + tx + 16 * b;
      if (qq >= nq) continue;
      int64_t ld;
      C* col = S.col(qq, ld);
#pragma unroll
      for (int a = 0; a < RM; ++a) {
        const int i = rt + ty * RM + a;
        if (i >= i1) continue;
        float lo, hi;
        asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[a][b]));
        C v = col[int64_t(i) * ld];
        v.x -= lo;
        v.y -= hi;
        col[int64_t(i) * ld] = v;
      }
    }
  } else {
    double ar[RM][RN], ai[RM][RN];
#pragma unroll
    for (int a = 0; a < RM; ++a)
#pragma unroll
      for (int b = 0; b < RN; ++b) ar[a][b] = ai[a][b] = 0.0;
    for (int k = 0; k < nb; ++k) {
      C p[RM], q[RN];
#pragma unroll
      for (int a = 0; a < RM; ++a) p[a] = Ps[(ty * RM + a) * LDP + k];
#pragma unroll
      for (int b = 0; b < RN; ++b) q[b] = Qs[k * TN + tx + 16 * b];
#pragma unroll
      for (int a = 0; a < RM; ++a)
#pragma unroll
        for (int b = 0; b < RN; ++b) cfma(ar[a][b], ai[a][b], double(p[a].x), double(p[a].y), double(q[b].x), double(q[b].y));
    }
#pragma unroll
    for (int b = 0; b < RN; ++b) {
      const int qq = qt + tx + 16 * b;
      if (qq >= nq) continue;
      int64_t ld;
      C* col = S.col(qq, ld);
#pragma unroll
      for (int a = 0; a < RM; ++a) {
        const int i = rt + ty * RM + a;
        if (i >= i1) continue;
        C v = col[int64_t(i) * ld];
        v.x -= ar[a][b];
        v.y -= ai[a][b];
        col[int64_t(i) * ld] = v;
      }
    }
  }
}

// ---------------------------------------------------------------- C += A B, complex64, C complex128, n x n
// 64 x 64 tiles of 256 threads, 16 columns of A and rows of B per step, the next step's
// entries loaded into registers while this one's are multiplied; packed FP32 pairs.
__global__ void __launch_bounds__(256) square_gemm_kernel(int n, const float2* __restrict__ A, const float2* __restrict__ B,
                                                          double2* __restrict__ C) {
  constexpr int TK = 16;
  __shared__ __align__(16) float2 As[64][TK + 2], Bs[TK][64];
  const int rt = blockIdx.y * 64, qt = blockIdx.x * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  unsigned long long acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0ull;
  float2 ra[4], rb[4];
  auto load = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = threadIdx.x + 256 * u;
      const int i = e / TK, k = e % TK, kb = e / 64, q = e % 64;
      ra[u] = rt + i < n && k0 + k < n ? A[int64_t(rt + i) * n + k0 + k] : make_float2(0.f, 0.f);
      rb[u] = k0 + kb < n && qt + q < n ? B[int64_t(k0 + kb) * n + qt + q] : make_float2(0.f, 0.f);
    }
  };
  load(0);
  for (int k0 = 0; k0 < n; k0 += TK) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = threadIdx.x + 256 * u;
      As[e / TK][e % TK] = ra[u];
      Bs[e / 64][e % 64] = rb[u];
    }
    __syncthreads();
    if (k0 + TK < n) load(k0 + TK);
#pragma unroll
    for (int k = 0; k < TK; k += 2) {
      float4 p[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) p[a] = *reinterpret_cast<const float4*>(&As[ty * 4 + a][k]);
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const float2 q0 = Bs[k][tx + 16 * b], q1 = Bs[k + 1][tx + 16 * b];
        const unsigned long long x0 = pk(q0.x, q0.y), y0 = pk(-q0.y, q0.x), x1 = pk(q1.x, q1.y), y1 = pk(-q1.y, q1.x);
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          fma2(acc[a][b], pk(p[a].x, p[a].x), x0);
          fma2(acc[a][b], pk(p[a].y, p[a].y), y0);
          fma2(acc[a][b], pk(p[a].z, p[a].z), x1);
          fma2(acc[a][b], pk(p[a].w, p[a].w), y1);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = rt + ty * 4 + a, q = qt + tx + 16 * b;
      if (i >= n || q >= n) continue;
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[a][b]));
      double2 v = C[int64_t(i) * n + q];
      v.x += widen(lo);
      v.y += widen(hi);
      C[int64_t(i) * n + q] = v;
    }
}

// ---------------------------------------------------------------- launches
// per function and context, shared by every launching thread: set once to the
// largest size a launch may ask for, never to one call's size
template <class K>
void allow_smem(K kernel, size_t bytes, std::atomic<uint64_t>& set, int dev) {
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (set.load() & bit) return;
  SLDM_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes)));
  set.fetch_or(bit);
}

template <class C, int TM, int TN>
void gemm_tile(const Cols<C>& S, const C* A, int n, int i0, int i1, int kc, int k0, int nb, int nq, const int* err, int dev,
               cudaStream_t s) {
  constexpr int NBW = panel_width<C>();
  constexpr size_t smem = (size_t(TM) * (NBW + 16 / sizeof(C)) + size_t(NBW) * TN) * sizeof(C);
  static std::atomic<uint64_t> set{0};
  allow_smem(lu_gemm_kernel<C, TM, TN>, smem, set, dev);
  lu_gemm_kernel<C, TM, TN><<<dim3((nq + TN - 1) / TN, (i1 - i0 + TM - 1) / TM), 256, smem, s>>>(S, A, n, i0, i1, kc, k0, nb, err),
      count_launch();
}
// tiles: the largest of which there are two for each SM
template <class C>
void lu_gemm(const Cols<C>& S, const C* A, int n, int i0, int i1, int kc, int k0, int nb, int nq, const int* err, int dev, int nsm,
             cudaStream_t s) {
  auto tiles = [&](int tm, int tn) { return int64_t((nq + tn - 1) / tn) * ((i1 - i0 + tm - 1) / tm); };
  if constexpr (sizeof(C) == 8) {
    if (tiles(128, 64) >= 2 * nsm) return gemm_tile<C, 128, 64>(S, A, n, i0, i1, kc, k0, nb, nq, err, dev, s);
  }
  if (tiles(64, 64) >= 2 * nsm) return gemm_tile<C, 64, 64>(S, A, n, i0, i1, kc, k0, nb, nq, err, dev, s);
  gemm_tile<C, 32, 32>(S, A, n, i0, i1, kc, k0, nb, nq, err, dev, s);
}

template <class C, int CS>
bool panel_cluster(C* A, int n, int j0, int nb, Moves* mv, int* err, int dev, cudaStream_t s) {
  constexpr size_t LIMIT = 200 * 1024;
  const int chunk = (n - j0 + CS - 1) / CS;
  const size_t smem = size_t(chunk) * (panel_width<C>() + 1) * sizeof(C);
  if (smem > LIMIT) return false;
  static ClusterFit fit;
  if (!cluster_fits(fit, dev, reinterpret_cast<const void*>(lu_panel_cluster<C, CS>), CS, PC_THREADS, LIMIT)) return false;
  ClusterLaunch c(CS, CS, PC_THREADS, smem, s);
  SLDM_CUDA(cudaLaunchKernelEx(&c.cfg, lu_panel_cluster<C, CS>, A, n, j0, nb, chunk, mv, err));
  count_launch();
  return true;
}

}  // namespace

void square_gemm_add(int n, const float2* A, const float2* B, double2* C, cudaStream_t s) {
  square_gemm_kernel<<<dim3((n + 63) / 64, (n + 63) / 64), 256, 0, s>>>(n, A, B, C), count_launch();
  SLDM_CUDA(cudaGetLastError());
}

template <class C>
void lu_solve_blocked(const LUSysT<C>& S, cudaStream_t s) {
  constexpr int NB = panel_width<C>();
  const int n = S.n, r = S.nrhs;
  int dev = 0, nsm = 0;
  SLDM_CUDA(cudaGetDevice(&dev));
  SLDM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  DBuf<int> piv, err;
  DBuf<Moves> mv;
  DBuf<C> urow, orow;
  DBuf<double> slot_v;
  DBuf<int> slot_i;
  DBuf<unsigned> bar;
  err.alloc(2);
  err.zero(s);
  mv.alloc(1);
  constexpr size_t solve_smem = (size_t(NB) * (NB + 1) + size_t(2) * NB * TS_COLS) * sizeof(C);
  static std::atomic<uint64_t> set_lo{0}, set_up{0}, set_panel{0};
  allow_smem(lu_solve_kernel<C, true>, solve_smem, set_lo, dev);
  allow_smem(lu_solve_kernel<C, false>, solve_smem, set_up, dev);
  // a panel taller than a cluster's shared memory: a cooperative launch over all SMs
  auto tall_panel = [&](int j0, int nb) {
    if (!piv.p) {
      piv.alloc(n);
      SLDM_CUDA(cudaMemsetAsync(piv.p, 0xff, size_t(n) * sizeof(int), s));  // -1: no pivot yet
      urow.alloc(NB);
      orow.alloc(NB);
      slot_v.alloc(nsm);
      slot_i.alloc(nsm);
      if (!bar.p) bar.alloc(1);
      const int max_chunk = (n + nsm - 1) / nsm > PANEL_MIN_ROWS ? (n + nsm - 1) / nsm : PANEL_MIN_ROWS;
      const size_t panel_smem = (size_t(max_chunk) * NB + NB) * sizeof(C);
      SLDM_REQUIRE(panel_smem <= 200 * 1024, SLDM_ENOTSUP, "LU: panel too large for shared memory");
      allow_smem(lu_panel_kernel<C>, 200 * 1024, set_panel, dev);
      int per_sm = 0;
      SLDM_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, lu_panel_kernel<C>, PANEL_THREADS, panel_smem));
      SLDM_REQUIRE(per_sm >= 1, SLDM_ENOTSUP, "LU: panel kernel does not fit on an SM");
    }
    const int rows = n - j0;
    const int G = std::max(1, std::min(nsm, (rows + PANEL_MIN_ROWS - 1) / PANEL_MIN_ROWS));
    const int chunk = (rows + G - 1) / G;
    SLDM_CUDA(cudaMemsetAsync(bar.p, 0, sizeof(unsigned), s));
    C* a0 = S.A;
    int a1 = n, a2 = j0, a3 = nb, a4 = chunk;
    int* a5 = piv.p;
    C* a6 = urow.p;
    C* a7 = orow.p;
    double* a8 = slot_v.p;
    int* a9 = slot_i.p;
    unsigned* a10 = bar.p;
    int* a11 = err.p;
    void* args[] = {&a0, &a1, &a2, &a3, &a4, &a5, &a6, &a7, &a8, &a9, &a10, &a11};
    const size_t sm = (size_t(chunk) * NB + NB) * sizeof(C);
    SLDM_CUDA(cudaLaunchCooperativeKernel((void*)lu_panel_kernel<C>, dim3(G), dim3(PANEL_THREADS), args, sm, s));
    count_launch();
    lu_moves_kernel<<<1, 32, 0, s>>>(piv.p, j0, nb, mv.p, err.p), count_launch();
  };
  ScopedTimer tm("lu_blocked", s);
  if (take_lu_stall()) {
    bar.alloc(1);
    bar.zero(s);
    lu_stall_kernel<<<1, 1, 0, s>>>(bar.p, err.p), count_launch();
  }
  for (int j0 = 0; j0 < n; j0 += NB) {
    const int nb = std::min(NB, n - j0);
    if (!panel_cluster<C, 16>(S.A, n, j0, nb, mv.p, err.p, dev, s) && !panel_cluster<C, 8>(S.A, n, j0, nb, mv.p, err.p, dev, s))
      tall_panel(j0, nb);
    Cols<C> R{S.A, n, j0 + nb, S.B, r};
    const int nq = (n - j0 - nb) + r;
    if (nq > 0) {
      lu_solve_kernel<C, true><<<(nq + TS_COLS - 1) / TS_COLS, TS_THREADS, solve_smem, s>>>(R, S.A, n, j0, nb, mv.p, err.p),
          count_launch();
      if (j0 + nb < n) lu_gemm<C>(R, S.A, n, j0 + nb, n, j0, j0, nb, nq, err.p, dev, nsm, s);
    }
    SLDM_CUDA(cudaGetLastError());
  }
  // back substitution U X = B on B's columns, panels from the bottom
  if (r > 0) {
    Cols<C> Bc{S.A, n, n, S.B, r};
    const int npan = (n + NB - 1) / NB;
    for (int p = npan - 1; p >= 0; --p) {
      const int j0 = p * NB, nb = std::min(NB, n - j0);
      lu_solve_kernel<C, false><<<(r + TS_COLS - 1) / TS_COLS, TS_THREADS, solve_smem, s>>>(Bc, S.A, n, j0, nb, nullptr, err.p),
          count_launch();
      if (j0 > 0) lu_gemm<C>(Bc, S.A, n, 0, j0, j0, j0, nb, r, err.p, dev, nsm, s);
    }
    SLDM_CUDA(cudaGetLastError());
  }
  int herr[2] = {0, 0};
  SLDM_CUDA(cudaMemcpyAsync(herr, err.p, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
  SLDM_CUDA(cudaStreamSynchronize(s));
  SLDM_REQUIRE(herr[0] != 2, SLDM_ETIMEOUT, "LU: a panel barrier ran out of its wait limit");
  SLDM_REQUIRE(herr[0] == 0, SLDM_ENUMERIC,
               "LU: zero or non-finite pivot in column " + std::to_string(herr[1]) + " of " + std::to_string(n));
}

template void lu_solve_blocked<float2>(const LUSysT<float2>&, cudaStream_t);
template void lu_solve_blocked<double2>(const LUSysT<double2>&, cudaStream_t);

}  // namespace sldm
