// Device helpers shared by the fill translation units: the 6-point rule,
// precision traits of the destination, FP64 closed-form potentials of a flat
// triangle, and the smooth remainders of G and grad G used on touching pairs.
#pragma once
#include <cmath>

#include "internal.h"

namespace sldm {

// ---------------------------------------------------------------- Dunavant rule
// Six-point degree-4 rule (Dunavant 1985): barycentric points and weights
// (weights sum to 1).
static __constant__ double c_bary[6][3] = {
    {0.108103018168070, 0.445948490915965, 0.445948490915965},
    {0.445948490915965, 0.108103018168070, 0.445948490915965},
    {0.445948490915965, 0.445948490915965, 0.108103018168070},
    {0.816847572980459, 0.091576213509771, 0.091576213509771},
    {0.091576213509771, 0.816847572980459, 0.091576213509771},
    {0.091576213509771, 0.091576213509771, 0.816847572980459}};
static __constant__ double c_w[6] = {0.223381589678011, 0.223381589678011, 0.223381589678011,
                              0.109951743655322, 0.109951743655322, 0.109951743655322};

constexpr double PI = 3.14159265358979323846;
constexpr double INV4PI = 0.25 / PI;

// ---------------------------------------------------------------- precision traits
template <class R>
struct M;
template <>
struct M<float> {
  // sin and cos of the FP32 phase k R: the argument is first reduced to
  // [-pi, pi] with 2 pi split into two floats (6.2831855 + (-1.7484555e-7), a
  // Cody-Waite reduction whose error stays below that of the FP32 argument
  // itself for |x| < 2^12), then the special-function unit evaluates sin and cos
  // (absolute error ~4e-7 on that interval).  Two SFU operations and five FMA-pipe
  // operations, against a long branchy sequence for sincosf: the bulk fill
  // inlines 36 of these per triangle pair.
  static __device__ __forceinline__ void sincos_(float x, float* s, float* c) {
    const float n = rintf(x * 0.15915494309189535f);
    const float r = __fmaf_rn(-n, -1.7484555e-7f, __fmaf_rn(-n, 6.2831855f, x));
    *s = __sinf(r);
    *c = __cosf(r);
  }
  static __device__ __forceinline__ float exp_(float x) { return __expf(x); }
  static __device__ __forceinline__ float rsqrt_(float x) { return rsqrtf(x); }
  static __device__ __forceinline__ void add(void* base, int64_t idx, float re, float im) {
    atomicAdd(reinterpret_cast<float2*>(base) + idx, make_float2(re, im));
  }
  static __device__ __forceinline__ void store(void* base, int64_t idx, double re, double im) {
    reinterpret_cast<float2*>(base)[idx] = make_float2(float(re), float(im));
  }
  static __device__ __forceinline__ void store_r(void* base, int64_t idx, float re, float im) {
    reinterpret_cast<float2*>(base)[idx] = make_float2(re, im);
  }
};
template <>
struct M<double> {
  static __device__ __forceinline__ void sincos_(double x, double* s, double* c) { sincos(x, s, c); }
  static __device__ __forceinline__ double exp_(double x) { return exp(x); }
  static __device__ __forceinline__ double rsqrt_(double x) { return rsqrt(x); }
  static __device__ __forceinline__ void add(void* base, int64_t idx, double re, double im) {
    double* p = reinterpret_cast<double*>(base) + 2 * idx;
    atomicAdd(p, re);
    atomicAdd(p + 1, im);
  }
  static __device__ __forceinline__ void store(void* base, int64_t idx, double re, double im) {
    reinterpret_cast<double2*>(base)[idx] = make_double2(re, im);
  }
  static __device__ __forceinline__ void store_r(void* base, int64_t idx, double re, double im) { store(base, idx, re, im); }
};
// atomic add of a double result into a destination of precision R
template <class R>
__device__ __forceinline__ void add_d(void* base, int64_t idx, double re, double im) {
  M<R>::add(base, idx, R(re), R(im));
}

// ---------------------------------------------------------------- FP64 kernel evaluations
// This part issues two FP64 operations per SM and clock (a warp instruction every
// 16 clocks) beside 128 FP32 or integer ones, so an FP64 fill costs what its FP64
// instructions cost.  exp(-j k R) therefore takes its argument in steps of a
// table, y = R (k 256 / 2 pi): the nearest step n and the remainder f = y - n come
// from adding and subtracting 1.5 2^52 (exact for |y| < 2^51), the table of the 256
// roots of unity lies in shared memory, and the remainder (an angle below
// pi / 256) needs three Taylor terms of sin and cos each to 1e-17:
// 14 FP64 operations, against ~35 of the general sincos, whose argument may have
// any size.  exp(Im k R) the same way from 256 powers of two (9 operations).
constexpr int WAVE_N = 256;
struct WaveTab {
  double2 cs[WAVE_N];  // (cos, sin)(2 pi i / 256)
  double ex[WAVE_N];   // 2^(i / 256)
};
// Fills the tables of a CTA (call with every thread, then __syncthreads).  The
// roots of one octant are computed, the others are their reflections.
__device__ __forceinline__ void wave_tab_fill(WaveTab& T, bool lossy) {
  for (int i = threadIdx.x; i <= WAVE_N / 8; i += blockDim.x) {
    double sn, cn;
    sincospi(double(i) / (WAVE_N / 2), &sn, &cn);
    T.cs[i] = make_double2(cn, sn);
    T.cs[64 - i] = make_double2(sn, cn);
    T.cs[64 + i] = make_double2(-sn, cn);
    T.cs[128 - i] = make_double2(-cn, sn);
    T.cs[128 + i] = make_double2(-cn, -sn);
    T.cs[192 - i] = make_double2(-sn, -cn);
    T.cs[192 + i] = make_double2(sn, -cn);
    T.cs[(WAVE_N - i) & (WAVE_N - 1)] = make_double2(cn, -sn);
  }
  if (lossy)
    for (int i = threadIdx.x; i < WAVE_N; i += blockDim.x) T.ex[i] = exp2(double(i) / WAVE_N);
}
static_assert(WAVE_N == 256, "octant reflections above");
// (cos, sin) of y steps of 2 pi / 256
__device__ __forceinline__ void wave_cis(const WaveTab& T, double y, double& c, double& s) {
  constexpr double H = 2.0 * PI / WAVE_N, H2 = H * H;
  const double t = __dadd_rn(y, 6755399441055744.0);
  const double f = __dsub_rn(y, __dsub_rn(t, 6755399441055744.0));
  const double2 w = T.cs[__double2loint(t) & (WAVE_N - 1)];
  const double f2 = f * f;
  const double sf = f * fma(f2, fma(f2, H * H2 * H2 / 120.0, -H * H2 / 6.0), H);
  const double cf = f2 * fma(f2, fma(f2, -H2 * H2 * H2 / 720.0, H2 * H2 / 24.0), -H2 / 2.0);  // cos - 1
  c = fma(-w.y, sf, fma(w.x, cf, w.x));
  s = fma(w.x, sf, fma(w.y, cf, w.y));
}
// 2^(y / 256); 0 or infinity where that leaves the normal range
__device__ __forceinline__ double wave_exp2(const WaveTab& T, double y) {
  constexpr double L = 0.69314718055994530942 / WAVE_N;
  const double t = __dadd_rn(y, 6755399441055744.0);
  const double f = __dsub_rn(y, __dsub_rn(t, 6755399441055744.0));
  const int n = __double2loint(t), yh = __double2hiint(y);
  const double w = T.ex[n & (WAVE_N - 1)];
  const double p = f * fma(f, fma(f, fma(f, L * L * L * L / 24.0, L * L * L / 6.0), L * L / 2.0), L);
  const double v = fma(w, p, w);
  int hi = __double2hiint(v) + ((n >> 8) << 20), lo = __double2loint(v);
  if ((yh & 0x7fffffff) >= 0x410fe800) {  // |y| >= 1021 x 256
    hi = yh < 0 ? 0 : 0x7ff00000;
    lo = 0;
  }
  return __hiloint2double(hi, lo);
}
// 1 / sqrt(x), x > 0: the special-function unit's 2^-20 estimate and one step of
// Householder's third-order iteration (error cubed: below the rounding)
__device__ __forceinline__ double rsqrt_pos(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(fma(e, 0.375, 0.5) * e, y, y);
}

// log2 of positive normal x from 128 values of log2 of the mantissa's leading bits and
// the series of the rest (|r| < 2^-7): ~11 FP64 operations, error a few 1e-17 + rounding
constexpr int LOG_N = 128;
struct LogTab {
  double2 t[LOG_N];  // (1 / c, log2 c), c the middle of [1 + i / 128, 1 + (i + 1) / 128)
};
__device__ __forceinline__ void log_tab_fill(LogTab& T) {
  for (int i = threadIdx.x; i < LOG_N; i += blockDim.x) {
    const double inv = 1.0 / (1.0 + (i + 0.5) / LOG_N);
    T.t[i] = make_double2(inv, -log2(inv));
  }
}
__device__ __forceinline__ double log2_pos(const LogTab& T, double x) {
  constexpr double L = 1.44269504088896340736;
  const int hi = __double2hiint(x);
  const double2 w = T.t[(hi >> 13) & (LOG_N - 1)];
  const double m = __hiloint2double((hi & 0x000fffff) | 0x3ff00000, __double2loint(x));
  const double r = fma(m, w.x, -1.0);
  const double p = r * fma(r, fma(r, fma(r, fma(r, fma(r, fma(r, L / 7.0, -L / 6.0), L / 5.0), -L / 4.0), L / 3.0), -L / 2.0), L);
  // the exponent as a double: 2^52 + 2^31 + e built from bits
  const double e = __dsub_rn(__hiloint2double(0x43300000, ((hi >> 20) - 1023) ^ int(0x80000000)), 4503601774854144.0);
  return (e + w.y) + p;
}
// 1 / x, x > 0: the special-function unit's 2^-20 estimate and one step of the hyperpower iteration of
// order three (Altman 1960), y (1 + e + e^2) with e = 1 - x y: the error cubed, below the rounding
__device__ __forceinline__ double recip_pos(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(fma(e, e, e), y, y);
}

__device__ __forceinline__ double bound_radius(const double* c, const double* p0, const double* p1, const double* p2) {
  double r = 0.0;
  const double* P[3] = {p0, p1, p2};
  for (int i = 0; i < 3; ++i) {
    const double dx = P[i][0] - c[0], dy = P[i][1] - c[1], dz = P[i][2] - c[2];
    r = fmax(r, sqrt(dx * dx + dy * dy + dz * dz));
  }
  return r;
}

// ---------------------------------------------------------------- contraction of a pair's moments
// N[u][v] = int int lambda_u lambda'_v kernel / (A A') holds all a pair needs: the local
// RWGs are s_i (r - V_i) / (2 A) with r = sum_u lambda_u V_u, so the areas cancel
// (factors s_i s_j / 4 remain: half_sign).  Vertices enter as a_i = c - V_i (GEO_AV).
template <class R>
__device__ __forceinline__ R half_sign(double sig) {  // on the sign bit: no FP64 compare
  return __double2hiint(sig) < 0 ? R(-0.5) : R(0.5);
}
template <class R>
__device__ __forceinline__ R sum9(const R (&n)[9]) {
  return ((n[0] + n[1]) + (n[2] + n[3])) + ((n[4] + n[5]) + (n[6] + n[7])) + n[8];
}
// put(i, j, value): sum_uv N_uv (V_u - V_i).(V'_v - V'_j) = T - P_i - Q_j + S D_ij, D_uv = V_u . V'_v,
// P_i = sum_v (sum_u N_uv) D_iv, Q_j = sum_u (sum_v N_uv) D_uj, T = sum N D
template <class R, class Put>
__device__ __forceinline__ void contract_L(const R (&Nr)[9], const R (&Ni)[9], R Sr, R Si, const R* av, const R* bv, Put put) {
  R D[9], Pr[3], Pi[3], Qr[3], Qi[3], Tr = 0, Ti = 0;
#pragma unroll
  for (int v = 0; v < 3; ++v)
#pragma unroll
    for (int u = 0; u < 3; ++u)
      D[3 * u + v] = av[3 * u] * bv[3 * v] + av[3 * u + 1] * bv[3 * v + 1] + av[3 * u + 2] * bv[3 * v + 2];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    Pr[i] = Pi[i] = Qr[i] = Qi[i] = R(0);
#pragma unroll
    for (int w = 0; w < 3; ++w) {
      Pr[i] += (Nr[w] + Nr[3 + w] + Nr[6 + w]) * D[3 * i + w];
      Pi[i] += (Ni[w] + Ni[3 + w] + Ni[6 + w]) * D[3 * i + w];
      Qr[i] += (Nr[3 * w] + Nr[3 * w + 1] + Nr[3 * w + 2]) * D[3 * w + i];
      Qi[i] += (Ni[3 * w] + Ni[3 * w + 1] + Ni[3 * w + 2]) * D[3 * w + i];
      Tr += Nr[3 * i + w] * D[3 * i + w];
      Ti += Ni[3 * i + w] * D[3 * i + w];
    }
  }
#pragma unroll
  for (int j = 0; j < 3; ++j)
#pragma unroll
    for (int i = 0; i < 3; ++i)
      put(i, j, (Tr - Pr[i]) - (Qr[j] - Sr * D[3 * i + j]), (Ti - Pi[i]) - (Qi[j] - Si * D[3 * i + j]));
}
// put(i, j, value): sum_uv N_uv (V_i - V'_j).((V'_v - V'_j) x (V_u - V_i)), the moments N of g1, from
// (r - V_i).((r - r') x (r' - V'_j)) = (V_i - V'_j).((r' - V'_j) x (r - V_i)).  With local vertices,
// dc = c - c', A = sum N V'_v, B = sum N V_u, X = sum N V'_v x V_u, S = sum N, q_ij = V_i x V'_j it is
// dc.X + V_i.X - V'_j.X - B.(dc x V'_j) - A.(V_i x dc) + (A - B - S dc).q_ij
template <class R, class Put>
__device__ __forceinline__ void contract_K(const R (&Nr)[9], const R (&Ni)[9], const R* av, const R* bv, const R* dc, Put put) {
  R Ar[3] = {0, 0, 0}, Ai[3] = {0, 0, 0}, Br[3] = {0, 0, 0}, Bi[3] = {0, 0, 0}, Xr[3] = {0, 0, 0}, Xi[3] = {0, 0, 0};
  R Sr = 0, Si = 0;
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    R cr[3], ci[3];  // sum_v N_uv b_v
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cr[d] = Nr[3 * u] * bv[d] + Nr[3 * u + 1] * bv[3 + d] + Nr[3 * u + 2] * bv[6 + d];
      ci[d] = Ni[3 * u] * bv[d] + Ni[3 * u + 1] * bv[3 + d] + Ni[3 * u + 2] * bv[6 + d];
      Ar[d] += cr[d];
      Ai[d] += ci[d];
    }
    const R rr = Nr[3 * u] + Nr[3 * u + 1] + Nr[3 * u + 2], ri = Ni[3 * u] + Ni[3 * u + 1] + Ni[3 * u + 2];
    Sr += rr;
    Si += ri;
    const R* a = av + 3 * u;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
      Br[d] += rr * a[d];
      Bi[d] += ri * a[d];
      Xr[d] += cr[d1] * a[d2] - cr[d2] * a[d1];
      Xi[d] += ci[d1] * a[d2] - ci[d2] * a[d1];
    }
  }
  // a, b have the opposite sign of V, V': A and B above hold -A and -B, X and q are even
  R Fr[3], Fi[3];  // A - B - S dc
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    Fr[d] = (Br[d] - Ar[d]) - Sr * dc[d];
    Fi[d] = (Bi[d] - Ai[d]) - Si * dc[d];
  }
  const R cxr = dc[0] * Xr[0] + dc[1] * Xr[1] + dc[2] * Xr[2], cxi = dc[0] * Xi[0] + dc[1] * Xi[1] + dc[2] * Xi[2];
  R hr[3], hi[3];  // the source's part
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const R bx = bv[3 * j], by = bv[3 * j + 1], bz = bv[3 * j + 2];
    const R px = dc[1] * bz - dc[2] * by, py = dc[2] * bx - dc[0] * bz, pz = dc[0] * by - dc[1] * bx;
    hr[j] = (bx * Xr[0] + by * Xr[1] + bz * Xr[2]) - (Br[0] * px + Br[1] * py + Br[2] * pz);
    hi[j] = (bx * Xi[0] + by * Xi[1] + bz * Xi[2]) - (Bi[0] * px + Bi[1] * py + Bi[2] * pz);
  }
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const R ax = av[3 * i], ay = av[3 * i + 1], az = av[3 * i + 2];
    const R px = ay * dc[2] - az * dc[1], py = az * dc[0] - ax * dc[2], pz = ax * dc[1] - ay * dc[0];
    const R tr = cxr - (ax * Xr[0] + ay * Xr[1] + az * Xr[2]) - (Ar[0] * px + Ar[1] * py + Ar[2] * pz);
    const R ti = cxi - (ax * Xi[0] + ay * Xi[1] + az * Xi[2]) - (Ai[0] * px + Ai[1] * py + Ai[2] * pz);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const R bx = bv[3 * j], by = bv[3 * j + 1], bz = bv[3 * j + 2];
      const R qx = ay * bz - az * by, qy = az * bx - ax * bz, qz = ax * by - ay * bx;
      put(i, j, tr + hr[j] + (Fr[0] * qx + Fr[1] * qy + Fr[2] * qz), ti + hi[j] + (Fi[0] * qx + Fi[1] * qy + Fi[2] * qz));
    }
  }
}

// ---------------------------------------------------------------- FP64 closed forms
// Integrals over the flat triangle (p1, p2, p3) seen from r: each surface
// integral is reduced to a sum over the three edges with the surface divergence
// theorem in the plane of the triangle (Wilton, Rao, Glisson, Schaubert, Al-Bundak
// and Butler, IEEE Trans. AP-32, 1984; Graglia, IEEE Trans. AP-41, 1993).
struct Pot {
  double inv_r, r;            // int 1/R, int R
  double por[3], pr[3];       // int (rho' - rho)/R, int (rho' - rho) R
  double grad[3];             // int grad_r (1/R)
  double rho[3];              // projection of r on the plane
};

static __device__ void potentials(const double* r, const double* p1, const double* p2, const double* p3, Pot& o) {
  double u[3], w[3], n[3];
  for (int d = 0; d < 3; ++d) {
    u[d] = p2[d] - p1[d];
    w[d] = p3[d] - p1[d];
  }
  n[0] = u[1] * w[2] - u[2] * w[1];
  n[1] = u[2] * w[0] - u[0] * w[2];
  n[2] = u[0] * w[1] - u[1] * w[0];
  double nn = sqrt(n[0] * n[0] + n[1] * n[1] + n[2] * n[2]);
  for (int d = 0; d < 3; ++d) n[d] /= nn;
  double h = n[0] * (r[0] - p1[0]) + n[1] * (r[1] - p1[1]) + n[2] * (r[2] - p1[2]);
  for (int d = 0; d < 3; ++d) o.rho[d] = r[d] - h * n[d];
  double ah = fabs(h);
  double sum_tf = 0, omega = 0, sum_r = 0;
  double por[3] = {0, 0, 0}, pr[3] = {0, 0, 0}, gm[3] = {0, 0, 0};
  const double* P[4] = {p1, p2, p3, p1};
  for (int e = 0; e < 3; ++e) {
    const double* a = P[e];
    const double* b = P[e + 1];
    double s[3], m[3];
    double L = sqrt((b[0] - a[0]) * (b[0] - a[0]) + (b[1] - a[1]) * (b[1] - a[1]) + (b[2] - a[2]) * (b[2] - a[2]));
    for (int d = 0; d < 3; ++d) s[d] = (b[d] - a[d]) / L;
    m[0] = s[1] * n[2] - s[2] * n[1];
    m[1] = s[2] * n[0] - s[0] * n[2];
    m[2] = s[0] * n[1] - s[1] * n[0];
    double sm = 0, sp = 0, t0 = 0;
    for (int d = 0; d < 3; ++d) {
      sm += (a[d] - o.rho[d]) * s[d];
      sp += (b[d] - o.rho[d]) * s[d];
      t0 += (a[d] - o.rho[d]) * m[d];
    }
    double R02 = t0 * t0 + h * h;
    double Rm = sqrt(sm * sm + R02), Rp = sqrt(sp * sp + R02);
    double f;
    if (sp <= 0 && sm <= 0) {
      f = log((Rm - sm) / (Rp - sp));
    } else {
      double num = sp > 0 ? Rp + sp : R02 / (Rp - sp);
      double den = sm > 0 ? Rm + sm : R02 / (Rm - sm);
      f = log(num / den);
    }
    double q1 = R02 + ah * Rp, q2 = R02 + ah * Rm;
    double beta = (q1 > 0 ? atan(t0 * sp / q1) : 0.0) - (q2 > 0 ? atan(t0 * sm / q2) : 0.0);
    omega += beta;
    sum_tf += t0 * f;
    double line1 = sp * Rp - sm * Rm + R02 * f;  // 2 int_edge R dl
    sum_r += t0 * line1;
    double line3 = (sp * Rp * Rp * Rp - sm * Rm * Rm * Rm) / 4.0 + 3.0 * R02 * (sp * Rp - sm * Rm) / 8.0 +
                   3.0 * R02 * R02 * f / 8.0;   // int_edge R^3 dl
    for (int d = 0; d < 3; ++d) {
      por[d] += m[d] * 0.5 * line1;
      pr[d] += m[d] * line3 / 3.0;
      gm[d] -= m[d] * f;
    }
  }
  o.inv_r = sum_tf - ah * omega;
  o.r = sum_r / 6.0 + h * h / 3.0 * o.inv_r;
  double sg = h > 0 ? 1.0 : (h < 0 ? -1.0 : 0.0);
  for (int d = 0; d < 3; ++d) {
    o.por[d] = por[d];
    o.pr[d] = pr[d];
    o.grad[d] = gm[d] - sg * omega * n[d];
  }
}

// complex helpers (double)
struct cd {
  double r, i;
};
__device__ __forceinline__ cd cmul(cd a, cd b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }

// G - 1/(4 pi R) + k^2 R/(8 pi) (Taylor series for |kR| < 0.05)
static __device__ cd green_smooth(cd k, double R) {
  cd x = {k.r * R, k.i * R};
  double ax = sqrt(x.r * x.r + x.i * x.i);
  if (ax < 0.05) {
    // sum_{n>=1, n!=2} (-j k)^n R^(n-1) / n!
    cd mjk = {k.i, -k.r};  // -j k
    cd p = mjk;            // (-jk)^1
    cd acc = p;            // n = 1 term (R^0)
    double Rp = 1.0, fact = 1.0;
    for (int n = 2; n <= 11; ++n) {
      p = cmul(p, mjk);
      Rp *= R;
      fact *= n;
      if (n == 2) continue;
      acc.r += p.r * Rp / fact;
      acc.i += p.i * Rp / fact;
    }
    return {acc.r * INV4PI, acc.i * INV4PI};
  }
  double sn, cn;
  sincos(x.r, &sn, &cn);
  double ex = exp(x.i);  // exp(-j k R) = exp(ki R) (cos - j sin)
  cd e = {ex * cn - 1.0, -ex * sn};
  cd k2 = cmul(k, k);
  return {e.r * INV4PI / R + k2.r * R * 0.5 * INV4PI, e.i * INV4PI / R + k2.i * R * 0.5 * INV4PI};
}

// g1 of grad(G - 1/(4 pi R)) = (r - r') g1: (1 - (1 + jkR) exp(-jkR)) / (4 pi R^3)
static __device__ cd grad_smooth(cd k, double R) {
  cd x = {-k.i * R, k.r * R};  // j k R
  double ax = sqrt(x.r * x.r + x.i * x.i);
  double iR3 = INV4PI / (R * R * R);
  if (ax < 0.05) {
    // sum_{n>=2} (-1)^n (n-1) x^n / n!
    cd p = x, acc = {0, 0};
    double fact = 1.0;
    for (int n = 2; n <= 13; ++n) {
      p = cmul(p, x);
      fact *= n;
      double c = ((n & 1) ? -1.0 : 1.0) * (n - 1) / fact;
      acc.r += c * p.r;
      acc.i += c * p.i;
    }
    return {acc.r * iR3, acc.i * iR3};
  }
  double sn, cn;
  sincos(k.r * R, &sn, &cn);
  double ex = exp(k.i * R);
  cd e = {ex * cn, -ex * sn};              // exp(-jkR)
  cd one_x = {1.0 + x.r, x.i};             // 1 + jkR
  cd pr = cmul(one_x, e);
  return {(1.0 - pr.r) * iR3, -pr.i * iR3};
}

// sum over the 8 lanes of a group
__device__ __forceinline__ double grp_sum8(double v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v;
}

}  // namespace sldm
