// Sparse block preconditioner P of Sec. III (Eq. pcext) and its analytic
// inverse through the Schur complement of the charge block:
//
//   P = [ diag L^A_m    diag I_x   D^T diag(L^phi_m) B       ]
//       [ diag mu L^A  -diag K     D^T diag(L^phi/eps) B     ]
//       [ F D           0          k0^2 I                    ]
//
// (row 2 carries -diag K, as the final system's row 2 carries -K).  With
// Lambda the per-edge inverse of the 2x2 block [[a, b], [c, d]] of diagonals,
// P x = r is solved by
//   S x3 = r3 - F D (L11 r1 + L12 r2),  S = k0^2 I - F D (L11 P13 + L12 P23),
//   [x1; x2] = Lambda ([r1; r2] - [P13; P23] x3).
// S is block diagonal by object (D, B, F are); each distinct block is formed on the
// device and inverted once per assembly: by the FP64 LU, from order SCHUR_REFINE_MIN on by a
// complex64 LU refined with FP64 residuals.
#include <algorithm>

#include "dense.h"
#include "pair32.cuh"
#include "precond.h"
#include "widen.cuh"

namespace sldm {

__device__ __forceinline__ double2 c_mul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 c_div(double2 a, double2 b) {
  double d = b.x * b.x + b.y * b.y;
  return make_double2((a.x * b.x + a.y * b.y) / d, (a.y * b.x - a.x * b.y) / d);
}
__device__ __forceinline__ double2 c_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 c_sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
template <class C>
__device__ __forceinline__ double2 ld2(const C* p, int64_t i) { return make_double2(double(p[i].x), double(p[i].y)); }

// per edge: Lambda = [[a, b], [c, d]]^-1 with a = L^A_m[m,m], b = I_x[m,m], c = (mu L^A)[m,m], d = -K[m,m]
template <class C>
__global__ void prec_edges_kernel(int ne, const int32_t* __restrict__ tplus, const int32_t* __restrict__ tri_obj,
                                  const PrecObj* __restrict__ objs, const C* __restrict__ LAm, const char* __restrict__ loc,
                                  const int32_t* __restrict__ ix_ptr, const int32_t* __restrict__ ix_col,
                                  const double* __restrict__ ix_val, double2* lam) {
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= ne) return;
  const PrecObj O = objs[tri_obj[tplus[m]]];
  const int ml = m - O.e0;
  const double2 a = ld2(LAm, int64_t(m) * ne + m);
  double bx = 0;
  for (int z = ix_ptr[m]; z < ix_ptr[m + 1]; ++z)
    if (ix_col[z] == m) bx = ix_val[z];
  const double2 b = make_double2(bx, 0.0);
  const C* LA = reinterpret_cast<const C*>(loc) + O.oLA;
  const C* K = reinterpret_cast<const C*>(loc) + O.oK;
  const double2 c = ld2(LA, int64_t(ml) * O.ne + ml);
  const double2 kd = ld2(K, int64_t(ml) * O.ne + ml);
  const double2 d = make_double2(-kd.x, -kd.y);
  const double2 det = c_sub(c_mul(a, d), c_mul(b, c));
  const double2 one = make_double2(1.0, 0.0);
  const double2 idet = c_div(one, det);
  lam[4 * m + 0] = c_mul(d, idet);
  lam[4 * m + 1] = c_mul(make_double2(-b.x, -b.y), idet);
  lam[4 * m + 2] = c_mul(make_double2(-c.x, -c.y), idet);
  lam[4 * m + 3] = c_mul(a, idet);
}

// per triangle: diagonals of L^phi_m (global) and of the object's L^phi/eps
template <class C>
__global__ void prec_tris_kernel(int nt, const int32_t* __restrict__ tri_obj, const PrecObj* __restrict__ objs,
                                 const C* __restrict__ LPm, const char* __restrict__ loc, double2* pdiag) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nt) return;
  const PrecObj O = objs[tri_obj[t]];
  const int tl = t - O.t0;
  const C* LP = reinterpret_cast<const C*>(loc) + O.oLP;
  pdiag[2 * t + 0] = ld2(LPm, int64_t(t) * nt + t);
  pdiag[2 * t + 1] = ld2(LP, int64_t(tl) * O.nt + tl);
}

// S_o[q, q2] = k0^2 delta - sum_{edges e of t(q)} D[t(q), e] (L11[e] P13[e, q2] + L12[e] P23[e, q2])
// P13[e, q2] = D[t(q2), e] pm[t(q2)] - D[last, e] pm[last]  (P23 with the object's diagonal)
// Writes S_o (row-major) and the identity right-hand side for its inversion.
__global__ void prec_schur_kernel(const PrecObj O, double k0, const int32_t* __restrict__ tri_edge,
                                  const int8_t* __restrict__ tri_sign, const int32_t* __restrict__ tplus,
                                  const int32_t* __restrict__ tminus, const double2* __restrict__ lam,
                                  const double2* __restrict__ pdiag, double2* S, double2* I) {
  const int nq = O.nt - 1;
  const int q2 = blockIdx.x * blockDim.x + threadIdx.x;
  const int q = blockIdx.y;
  if (q2 >= nq) return;
  const int t = O.t0 + q, t2 = O.t0 + q2, last = O.t0 + O.nt - 1;
  double2 acc = make_double2(q == q2 ? k0 * k0 : 0.0, 0.0);
  for (int i = 0; i < 3; ++i) {
    const int e = tri_edge[3 * t + i];
    const double s = double(tri_sign[3 * t + i]);  // D[t, e]
    const double d2 = (tplus[e] == t2) ? 1.0 : ((tminus[e] == t2) ? -1.0 : 0.0);
    const double dl = (tplus[e] == last) ? 1.0 : ((tminus[e] == last) ? -1.0 : 0.0);
    if (d2 == 0.0 && dl == 0.0) continue;
    const double2 p13 = c_sub(make_double2(d2 * pdiag[2 * t2].x, d2 * pdiag[2 * t2].y),
                              make_double2(dl * pdiag[2 * last].x, dl * pdiag[2 * last].y));
    const double2 p23 = c_sub(make_double2(d2 * pdiag[2 * t2 + 1].x, d2 * pdiag[2 * t2 + 1].y),
                              make_double2(dl * pdiag[2 * last + 1].x, dl * pdiag[2 * last + 1].y));
    const double2 v = c_add(c_mul(lam[4 * e + 0], p13), c_mul(lam[4 * e + 1], p23));
    acc.x -= s * v.x;
    acc.y -= s * v.y;
  }
  S[int64_t(q) * nq + q2] = acc;
  I[int64_t(q) * nq + q2] = make_double2(q == q2 ? 1.0 : 0.0, 0.0);
}

template <class CV>
__device__ __forceinline__ CV to_cv(double2 v);
template <>
__device__ __forceinline__ double2 to_cv<double2>(double2 v) { return v; }
template <>
__device__ __forceinline__ float2 to_cv<float2>(double2 v) { return make_float2(float(v.x), float(v.y)); }
template <class CX>
__device__ __forceinline__ double2 wide2(const CX v) { return make_double2(widen(v.x), widen(v.y)); }

// t3 = s3 r3 - F D (L11 r1 + L12 r2) (per charge unknown; column blockIdx.y).  Complex64 columns in
// pairs of FP32 (pair32.cuh), the coefficients held as pairs; in FP64 this kernel and the next were bound by its pipe
// (N = 34,524, 32 columns: 26 -> 8 us and 39 -> 9 us).
template <class CX, class CV>
__global__ void prec_apply1_kernel(int ne, int nq, const int32_t* __restrict__ q2t, const int32_t* __restrict__ tri_edge,
                                   const int8_t* __restrict__ tri_sign, const double2* __restrict__ lam,
                                   const float4* __restrict__ lam32, VecBatch<CX, double2> rb, double s3, float2 s3f, CV* t3) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const CX* __restrict__ r = rb.x[blockIdx.y];
  const int t = q2t[q];
  if constexpr (sizeof(CX) == sizeof(float2)) {  // in pairs of FP32
    P32 re, im;
    const CX r3 = r[2 * ne + q];
    re.fma(s3f.x, s3f.y, r3.x);
    im.fma(s3f.x, s3f.y, r3.y);
    for (int i = 0; i < 3; ++i) {
      const int e = tri_edge[3 * t + i];
      const float sg = tri_sign[3 * t + i] < 0 ? 1.f : -1.f;
      const CX u = r[e], v = r[ne + e];
      cfma_pair(re, im, lam32[4 * e], sg * u.x, sg * u.y);
      cfma_pair(re, im, lam32[4 * e + 1], sg * v.x, sg * v.y);
    }
    CV o;
    re.get(o.x);
    im.get(o.y);
    t3[int64_t(blockIdx.y) * nq + q] = o;
    return;
  }
  double2 acc = wide2(r[2 * ne + q]);
  acc.x *= s3;
  acc.y *= s3;
  for (int i = 0; i < 3; ++i) {
    const int e = tri_edge[3 * t + i];
    const double2 v = c_add(c_mul(lam[4 * e + 0], wide2(r[e])), c_mul(lam[4 * e + 1], wide2(r[ne + e])));
    const bool neg = tri_sign[3 * t + i] < 0;
    acc.x += neg ? v.x : -v.x;
    acc.y += neg ? v.y : -v.y;
  }
  t3[int64_t(blockIdx.y) * nq + q] = to_cv<CV>(acc);
}

// x1, x2 = Lambda (r1 - P13 x3, r2 - P23 x3) and x3, with bx = B x3 (column blockIdx.y).
// WORK: into the product's work vectors; else added to the columns rb.y.
struct PrecWork {
  void *j, *a, *e, *bu, *bc;
};
template <class CX, class CV, bool WORK>
__global__ void __launch_bounds__(128) prec_apply45_kernel(int ne, int nq, int nt, const int32_t* __restrict__ tplus,
                                                           const int32_t* __restrict__ tminus, const int32_t* __restrict__ q2t,
                                                           const double2* __restrict__ lam, const double2* __restrict__ pdiag,
                                                           const float4* __restrict__ lam32, const float4* __restrict__ pdiag32,
                                                           VecBatch<CX, double2> rb, const CV* __restrict__ bx, PrecWork W) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t c = blockIdx.y;
  const CX* __restrict__ r = rb.x[c];
  bx += c * nt;
  if constexpr (WORK && sizeof(CX) == sizeof(float2)) {  // in pairs of FP32
    if (i < ne) {
      const int tp = tplus[i], tm = tminus[i];
      const CV bp = bx[tp], bm = bx[tm];
      P32 yr[2], yi[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const CX rk = r[k * ne + i];
        yr[k].add(rk.x);
        yi[k].add(rk.y);
        cfma_pair(yr[k], yi[k], pdiag32[2 * tp + k], -bp.x, -bp.y);
        cfma_pair(yr[k], yi[k], pdiag32[2 * tm + k], bm.x, bm.y);
      }
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        P32 xr, xi;
        cfma_pair(xr, xi, lam32[4 * i + 2 * k], yr[0], yi[0]);
        cfma_pair(xr, xi, lam32[4 * i + 2 * k + 1], yr[1], yi[1]);
        CV v;
        xr.get(v.x);
        xi.get(v.y);
        if (k == 0) {
          reinterpret_cast<CV*>(W.j)[c * ne + i] = v;
          reinterpret_cast<CV*>(W.a)[c * ne + i] = v;
        } else {
          reinterpret_cast<CV*>(W.e)[c * ne + i] = v;
        }
      }
    }
  } else if (i < ne) {
    const int tp = tplus[i], tm = tminus[i];
    const double2 bp = wide2(bx[tp]), bm = wide2(bx[tm]);
    const double2 y1 = c_sub(wide2(r[i]), c_sub(c_mul(pdiag[2 * tp], bp), c_mul(pdiag[2 * tm], bm)));
    const double2 y2 = c_sub(wide2(r[ne + i]), c_sub(c_mul(pdiag[2 * tp + 1], bp), c_mul(pdiag[2 * tm + 1], bm)));
    const double2 x1 = c_add(c_mul(lam[4 * i + 0], y1), c_mul(lam[4 * i + 1], y2));
    const double2 x2 = c_add(c_mul(lam[4 * i + 2], y1), c_mul(lam[4 * i + 3], y2));
    if (WORK) {
      const CV v = to_cv<CV>(x1);
      reinterpret_cast<CV*>(W.j)[c * ne + i] = v;
      reinterpret_cast<CV*>(W.a)[c * ne + i] = v;
      reinterpret_cast<CV*>(W.e)[c * ne + i] = to_cv<CV>(x2);
    } else {
      double2* xc = rb.y[c];
      xc[i] = c_add(xc[i], x1);
      xc[ne + i] = c_add(xc[ne + i], x2);
    }
  }
  if (WORK) {
    if (i < nt) {
      const CV v = bx[i];
      reinterpret_cast<CV*>(W.bu)[c * nt + i] = v;
      reinterpret_cast<CV*>(W.bc)[c * nt + i] = v;
    }
  } else if (i < nq) {
    double2* xc = rb.y[c] + 2 * ne;
    xc[i] = c_add(xc[i], wide2(bx[q2t[i]]));
  }
}

__global__ void split_c_kernel(int64_t n, const double2* __restrict__ a, float4* b) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float x = float(a[i].x), y = float(a[i].y);
  b[i] = make_float4(x, y, float(a[i].x - double(x)), float(a[i].y - double(y)));
}
__global__ void to_c64_kernel(int64_t n, const double2* __restrict__ a, float2* b) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    b[i] = make_float2(float(a[i].x), float(a[i].y));
}

// ---------------------------------------------------------------- inverse of a large Schur complement
// S is sparse up to the eliminated charge: S X = k0^2 X - G (B X) with G's row of triangle t
// holding t and its three neighbours, so I - S X costs 20 FP64 operations per entry where the
// factorisation costs 8/3 n of them.  X = S^-1 therefore starts from the complex64 inverse X32
// (blocked LU) and is refined, X += X32 (I - S X) with the bracket in FP64 and the
// product in FP32, each step gaining the digits X32 has, until I - S X is at the rounding of
// its own terms (FP64 operators) or below what the rounding of the stored inverse to complex64
// leaves (the others).
struct SchurRow {
  int32_t t[4];   // local triangles: itself, the neighbours across its edges
  double2 g[4];
};
__global__ void schur_rows_kernel(const PrecObj O, const int32_t* __restrict__ tri_edge, const int32_t* __restrict__ tplus,
                                  const int32_t* __restrict__ tminus, const double2* __restrict__ lam,
                                  const double2* __restrict__ pdiag, SchurRow* rows) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= O.nt - 1) return;
  const int t = O.t0 + q;
  SchurRow R;
  R.t[0] = q;
  R.g[0] = make_double2(0.0, 0.0);
  for (int i = 0; i < 3; ++i) {
    const int e = tri_edge[3 * t + i], n = tplus[e] == t ? tminus[e] : tplus[e];
    R.g[0] = c_add(R.g[0], c_add(c_mul(lam[4 * e], pdiag[2 * t]), c_mul(lam[4 * e + 1], pdiag[2 * t + 1])));
    const double2 v = c_add(c_mul(lam[4 * e], pdiag[2 * n]), c_mul(lam[4 * e + 1], pdiag[2 * n + 1]));
    R.t[1 + i] = n - O.t0;
    R.g[1 + i] = make_double2(-v.x, -v.y);
  }
  rows[q] = R;
}
// E = I - S X (rounded to complex64; X: nq + 1 rows, the last minus the sum of the others);
// emax[0] = its largest |Re|, |Im|, emax[1] = that of its terms, as float bits
__global__ void __launch_bounds__(128) schur_residual_kernel(int nq, double k02, const SchurRow* __restrict__ rows,
                                                             const double2* __restrict__ X, float2* __restrict__ E, unsigned* emax) {
  const int c = blockIdx.x * 128 + threadIdx.x, q = blockIdx.y;
  float m = 0.f, t = 0.f;
  if (c < nq) {
    const double2 x = X[int64_t(q) * nq + c];
    double er = (q == c ? 1.0 : 0.0) - k02 * x.x, ei = -k02 * x.y;
    t = float(fabs(er) + fabs(ei));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double2 g = rows[q].g[i], y = X[int64_t(rows[q].t[i]) * nq + c];
      t = fmaxf(t, (fabsf(float(g.x)) + fabsf(float(g.y))) * (fabsf(float(y.x)) + fabsf(float(y.y))));
      er = fma(g.x, y.x, fma(-g.y, y.y, er));
      ei = fma(g.x, y.y, fma(g.y, y.x, ei));
    }
    E[int64_t(q) * nq + c] = make_float2(float(er), float(ei));
    m = fmaxf(fabsf(float(er)), fabsf(float(ei)));
    if (!(m < 1e30f)) m = 1e30f;  // NaN too
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    t = fmaxf(t, __shfl_xor_sync(0xffffffffu, t, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(emax, __float_as_uint(m));
    atomicMax(emax + 1, __float_as_uint(t));
  }
}
// X's last row: minus the sum of the n others, with compensated sums (their rounding is what
// limits |I - S X|).  32 columns x 32 row groups per CTA.
__device__ __forceinline__ void two_sum(double& s, double& c, double v) {
  const double t = s + v, b = t - s;
  c += (s - (t - b)) + (v - b);
  s = t;
}
__global__ void __launch_bounds__(1024) last_row_kernel(int n, double2* X) {
  __shared__ double red[4][32][33];
  const int cx = threadIdx.x & 31, g = threadIdx.x >> 5, col = blockIdx.x * 32 + cx;
  double s[4] = {0, 0, 0, 0};  // re, its error, im, its error
  if (col < n)
#pragma unroll 4
    for (int r = g; r < n; r += 32) {
      const double2 v = X[int64_t(r) * n + col];
      two_sum(s[0], s[1], v.x);
      two_sum(s[2], s[3], v.y);
    }
  for (int i = 0; i < 4; ++i) red[i][g][cx] = s[i];
  __syncthreads();
  if (g != 0 || col >= n) return;
  for (int q = 1; q < 32; ++q)
    for (int i = 0; i < 4; i += 2) {
      two_sum(s[i], s[i + 1], red[i][q][cx]);
      s[i + 1] += red[i + 1][q][cx];
    }
  X[int64_t(n) * n + col] = make_double2(-(s[0] + s[1]), -(s[2] + s[3]));
}
__global__ void to_c128_kernel(int64_t n, const float2* __restrict__ a, double2* b) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) b[i] = make_double2(widen(a[i].x), widen(a[i].y));
}
__global__ void identity_c64_kernel(int n, float2* b) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;  // n x n
  if (i < int64_t(n) * n) b[i] = make_float2(i / n == i % n ? 1.f : 0.f, 0.f);
}

// X (nq + 1 rows) = B S^-1; false when the refinement does not converge (S is then intact).
// Whole assemblies with the FP64 LU and so, from the line on (smaller systems are one launch of the
// batched LU): sphere of 320 triangles, complex128 19.5 -> 18.6 ms, complex64 8.8 -> 7.7; box of 892,
// 152 -> 144 and 32.3 -> 23.5; of 1,356, 167 -> 142 and 69 -> 43.
constexpr int SCHUR_REFINE_MIN = 256;
static bool schur_inverse(const PrecObj& O, const DevMesh& d, const Precond& P, double k0, const double2* S, double2* X,
                          float goal, cudaStream_t s) {
  const int nq = O.nt - 1;
  const int64_t nn = int64_t(nq) * nq;
  const unsigned blocks = unsigned((nn + 255) / 256);
  DBuf<float2> A, X32;  // A: the factors, then I - S X
  DBuf<SchurRow> rows;
  DBuf<unsigned> emax;
  A.alloc(nn);
  X32.alloc(nn);
  rows.alloc(nq);
  emax.alloc(2);
  to_c64_kernel<<<std::min<int64_t>((nn + 255) / 256, 4096), 256, 0, s>>>(nn, S, A.p), ::sldm::count_launch();
  identity_c64_kernel<<<blocks, 256, 0, s>>>(nq, X32.p), ::sldm::count_launch();
  schur_rows_kernel<<<(nq + 127) / 128, 128, 0, s>>>(O, d.tri_edge.p, d.tplus.p, d.tminus.p, P.lam.p, P.pdiag.p, rows.p),
      ::sldm::count_launch();
  lu_solve_blocked<float2>(LUSysT<float2>{A.p, X32.p, nq, nq}, s);
  to_c128_kernel<<<blocks, 256, 0, s>>>(nn, X32.p, X), ::sldm::count_launch();
  float prev = 1e30f;
  for (int it = 0; it < 12; ++it) {
    last_row_kernel<<<(nq + 31) / 32, 1024, 0, s>>>(nq, X), ::sldm::count_launch();
    emax.zero(s);
    schur_residual_kernel<<<dim3((nq + 127) / 128, nq), 128, 0, s>>>(nq, k0 * k0, rows.p, X, A.p, emax.p), ::sldm::count_launch();
    SLDM_CUDA(cudaGetLastError());
    float em[2];
    SLDM_CUDA(cudaMemcpyAsync(em, emax.p, sizeof(em), cudaMemcpyDeviceToHost, s));
    SLDM_CUDA(cudaStreamSynchronize(s));
    const float e = em[0];
    const float ulp = 2.2e-16f * em[1];  // rounding of the terms
    if (!(em[1] < 1e30f && e < 0.5f)) return false;
    if (e <= std::max(goal, 4.f * ulp)) return true;
    // no longer falling: at its rounding, or not converging.  |I - S X| ends at 1 to 23 of these units (spheres, boxes,
    // wires of order 319 to 2,047), the FP64 LU's at 4 to 930
    if (!(e <= 0.25f * prev)) return e <= 64.f * ulp;
    prev = e;
    square_gemm_add(nq, X32.p, A.p, X, s);
  }
  return false;
}

template <class C>
void prec_setup(Precond& P, const sldm_mesh* m, const std::vector<PrecObj>& objs, double k0, const void* LAm,
                const void* LPm, const char* loc, const double* ix_val, cudaStream_t s) {
  const HostMesh& h = m->h;
  const DevMesh& d = m->d;
  const int ne = int(h.ne), nt = int(h.nt);
  P.objs.upload(objs, s);
  P.lam.alloc(size_t(4) * ne);
  P.pdiag.alloc(size_t(2) * nt);
  prec_edges_kernel<C><<<(ne + 127) / 128, 128, 0, s>>>(ne, d.tplus.p, d.obj.p, P.objs.p, (const C*)LAm, loc, d.ix_ptr.p,
                                                        d.ix_col.p, ix_val, P.lam.p), ::sldm::count_launch();
  prec_tris_kernel<C><<<(nt + 127) / 128, 128, 0, s>>>(nt, d.obj.p, P.objs.p, (const C*)LPm, loc, P.pdiag.p), ::sldm::count_launch();
  SLDM_CUDA(cudaGetLastError());
  // one block for each distinct Schur complement; repeated objects share it
  int64_t tot = 0, stot = 0;
  std::vector<int64_t> off(objs.size()), soff(objs.size());
  for (size_t i = 0; i < objs.size(); ++i) {
    const int64_t nq = objs[i].nt - 1;
    if (objs[i].same != int(i)) {
      off[i] = off[objs[i].same];
      continue;
    }
    off[i] = tot;
    soff[i] = stot;
    tot += (nq + 1) * nq;
    stot += nq * nq;
  }
  DBuf<double2> Sm;
  Sm.alloc(stot);
  P.sinv.alloc(tot);
  // of a complex64 operator the inverse is kept as complex64: |I - S X| <= 2^-33, n of which add up
  // to X's error, stays below that rounding for n up to ~10^4 (random signs)
  const float goal = sizeof(C) == sizeof(float2) ? 0x1p-33f : 0.f;
  std::vector<LUSys> sys;
  for (size_t i = 0; i < objs.size(); ++i) {
    const PrecObj& o = objs[i];
    if (o.same != int(i)) continue;
    const int nq = o.nt - 1;
    prec_schur_kernel<<<dim3((nq + 127) / 128, nq), 128, 0, s>>>(o, k0, d.tri_edge.p, d.tri_sign.p, d.tplus.p, d.tminus.p,
                                                                P.lam.p, P.pdiag.p, Sm.p + soff[i], P.sinv.p + off[i]), ::sldm::count_launch();
    if (nq >= SCHUR_REFINE_MIN) {
      bool done = false;
      try {
        done = schur_inverse(o, d, P, k0, Sm.p + soff[i], P.sinv.p + off[i], goal, s);
      } catch (const Error& e) {  // a pivot that FP32 loses, or no room beside the operator: in FP64, in place
        if (e.code != SLDM_ENUMERIC && e.code != SLDM_ENOMEM) throw;
      }
      if (done) continue;
      prec_schur_kernel<<<dim3((nq + 127) / 128, nq), 128, 0, s>>>(o, k0, d.tri_edge.p, d.tri_sign.p, d.tplus.p, d.tminus.p,
                                                                  P.lam.p, P.pdiag.p, Sm.p + soff[i], P.sinv.p + off[i]), ::sldm::count_launch();
    }
    sys.push_back({Sm.p + soff[i], P.sinv.p + off[i], nq, nq});
  }
  SLDM_CUDA(cudaGetLastError());
  lu_solve_batched(sys, s);  // sinv <- S^-1
  for (size_t i = 0; i < objs.size(); ++i)
    if (objs[i].same == int(i) && objs[i].nt > 1)
      last_row_kernel<<<(objs[i].nt + 30) / 32, 1024, 0, s>>>(objs[i].nt - 1, P.sinv.p + off[i]), ::sldm::count_launch();
  // a complex64 operator takes an FP32 preconditioner: S^-1 (accurate beyond
  // that rounding) in complex64, applied with FP32 arithmetic
  P.f32 = sizeof(C) == sizeof(float2);
  if (P.f32) {
    P.lam32.alloc(size_t(4) * ne);
    P.pdiag32.alloc(size_t(2) * nt);
    split_c_kernel<<<(4 * ne + 255) / 256, 256, 0, s>>>(4 * ne, P.lam.p, P.lam32.p), ::sldm::count_launch();
    split_c_kernel<<<(2 * nt + 255) / 256, 256, 0, s>>>(2 * nt, P.pdiag.p, P.pdiag32.p), ::sldm::count_launch();
  }
  if (P.f32 && tot > 0) {
    P.sinv32.alloc(tot);
    to_c64_kernel<<<std::min<int64_t>((tot + 255) / 256, 4096), 256, 0, s>>>(tot, P.sinv.p, P.sinv32.p), ::sldm::count_launch();
    SLDM_CUDA(cudaGetLastError());
    SLDM_CUDA(cudaStreamSynchronize(s));
    P.sinv.release();
  }
  // GEMV plan: (B x3)_o = B_o S_o^-1 t3_o, WR columns
  const size_t ev = P.f32 ? sizeof(float2) : sizeof(double2);
  P.nq = h.nt - h.nobj;
  const int64_t nq1 = std::max<int64_t>(P.nq, 1);
  P.t3.alloc(nq1 * MAX_NRHS);
  P.bx.alloc(h.nt * MAX_NRHS);
  std::vector<GemvJob> jobs;
  std::vector<int64_t> rs;
  std::vector<int2> tiles;
  int64_t acc = 0;
  const char* A0 = P.f32 ? (const char*)P.sinv32.p : (const char*)P.sinv.p;
  for (size_t i = 0; i < objs.size(); ++i) {
    const int nq = objs[i].nt - 1;
    if (nq <= 0) continue;
    for (int r0 = 0; r0 < nq + 1; r0 += gemv_tile_rows(ev)) tiles.push_back(make_int2(int(jobs.size()), r0));
    jobs.push_back({A0 + off[i] * ev, nq, nq + 1, nq, (char*)P.t3.p + objs[i].q0 * ev, P.nq, (char*)P.bx.p + objs[i].t0 * ev,
                    h.nt, 1, 0, 0, 0});
    rs.push_back(acc);
    acc += nq + 1;
  }
  P.jobs.upload(jobs, s);
  P.rs.upload(rs, s);
  P.tiles.upload(tiles, s);
  P.plan.jobs = P.jobs.p;
  P.plan.rowstart = P.rs.p;
  P.plan.njobs = int(jobs.size());
  P.plan.total_rows = acc;
  P.plan.tiles = P.tiles.p;
  P.plan.ntiles = int(tiles.size());
  P.plan.tile_rows = gemv_tile_rows(ev);
  P.plan.name = "gemv_pc";
  P.plan.bytes = 0;
  for (auto& jb : jobs) P.plan.bytes += double(jb.m) * jb.n * ev;
  P.plan.tc = nullptr;
  if (P.f32) {
    tc_plan_build(jobs, P.tc, true, s);
    if (P.tc.ok) P.plan.tc = &P.tc;
  }
  SLDM_CUDA(cudaStreamSynchronize(s));
}

// B x3 of every column: the right-hand side of the Schur complement and its inverse
template <class CX, class CV>
static void prec_charges(const Precond& P, const sldm_mesh* m, const VecBatch<CX, double2>& r, double s3, int nr,
                         cudaStream_t s) {
  SLDM_REQUIRE((nr >= 1 && nr <= MAX_NRHS), SLDM_EINVAL, "preconditioner: 1 to 32 columns");
  const DevMesh& d = m->d;
  const int ne = int(m->h.ne), nq = int(P.nq);
  prec_apply1_kernel<CX, CV><<<dim3((nq + 127) / 128, nr), 128, 0, s>>>(ne, nq, d.q2t.p, d.tri_edge.p, d.tri_sign.p, P.lam.p,
                                                                      P.lam32.p, r, s3, make_float2(float(s3), float(s3 - double(float(s3)))),
                                                                      reinterpret_cast<CV*>(P.t3.p)), ::sldm::count_launch();
  gemv_jobs<CV>(P.plan, nr, s);
}

template <class CX, class C>
void prec_apply_in(const Precond& P, const sldm_mesh* m, const VecBatch<CX, double2>& r, double s3, void* j, void* a, void* e,
                   void* bu, void* bc, int nr, cudaStream_t s) {
  ScopedTimer tm("precond", s);
  const DevMesh& d = m->d;
  const int ne = int(m->h.ne), nq = int(P.nq), nt = int(m->h.nt);
  prec_charges<CX, C>(P, m, r, s3, nr, s);
  prec_apply45_kernel<CX, C, true><<<dim3((std::max(ne, nt) + 127) / 128, nr), 128, 0, s>>>(
      ne, nq, nt, d.tplus.p, d.tminus.p, d.q2t.p, P.lam.p, P.pdiag.p, P.lam32.p, P.pdiag32.p, r, reinterpret_cast<const C*>(P.bx.p),
      PrecWork{j, a, e, bu, bc}), ::sldm::count_launch();
  SLDM_CUDA(cudaGetLastError());
}
template void prec_apply_in<float2, float2>(const Precond&, const sldm_mesh*, const VecBatch<float2, double2>&, double, void*,
                                            void*, void*, void*, void*, int, cudaStream_t);
template void prec_apply_in<double2, double2>(const Precond&, const sldm_mesh*, const VecBatch<double2, double2>&, double, void*,
                                              void*, void*, void*, void*, int, cudaStream_t);

template <class CV>
static void prec_add_t(const Precond& P, const sldm_mesh* m, const VecBatch<double2, double2>& r, double s3, int nr,
                       cudaStream_t s) {
  const DevMesh& d = m->d;
  const int ne = int(m->h.ne), nq = int(P.nq), nt = int(m->h.nt);
  prec_charges<double2, CV>(P, m, r, s3, nr, s);
  prec_apply45_kernel<double2, CV, false><<<dim3((std::max(ne, nt) + 127) / 128, nr), 128, 0, s>>>(
      ne, nq, nt, d.tplus.p, d.tminus.p, d.q2t.p, P.lam.p, P.pdiag.p, P.lam32.p, P.pdiag32.p, r, reinterpret_cast<const CV*>(P.bx.p), PrecWork{}),
      ::sldm::count_launch();
  SLDM_CUDA(cudaGetLastError());
}
void prec_apply_add(const Precond& P, const sldm_mesh* m, const VecBatch<double2, double2>& r, double s3, int nr,
                    cudaStream_t s) {
  ScopedTimer tm("precond", s);
  if (P.f32) prec_add_t<float2>(P, m, r, s3, nr, s);
  else prec_add_t<double2>(P, m, r, s3, nr, s);
}

template void prec_setup<float2>(Precond&, const sldm_mesh*, const std::vector<PrecObj>&, double, const void*, const void*,
                                 const char*, const double*, cudaStream_t);
template void prec_setup<double2>(Precond&, const sldm_mesh*, const std::vector<PrecObj>&, double, const void*, const void*,
                                  const char*, const double*, cudaStream_t);

}  // namespace sldm
