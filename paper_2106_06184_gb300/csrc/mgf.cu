// Layered-medium Green's function of the external problem (Sec. II-C; Sec. IV:
// quasistatic part extracted and added back analytically, Sommerfeld integrals
// of the rest tabulated and interpolated), for source and observation points in
// one layer l of a stratified background.
//
// Mixed-potential kernels (normalised like the paper's operators: L^A_m uses
// G^A/mu0, L^phi_m uses eps0 K^phi), spectral form from transmission-line
// Green's functions of the TM (e) and TE (h) lines of layer l:
//   g_xx = V_i^h/(j w mu0),  k_phi = eps0 (j w/k_rho^2)(V_i^e - V_i^h),
//   g_zz = [mu_r (k_rho^2 - k_z^2)/(eps k_rho^2) I_v^e + (w^2 mu mu_r/k_rho^2) I_v^h]/(j w),
//   g_zu = j (mu_r/k_rho)(I_i^e - I_i^h),  g_uz = j (mu_r/k_rho)(V_v^e - V_v^h),
// spatial: S0 for xx, phi, zz and -j S1 for z-rho, rho-z (S_n[f] = 1/(2 pi) int f J_n k dk).
// The direct term (homogeneous kernel of layer l) is filled by the homogeneous
// path; the quasistatic images of the two adjacent interfaces are evaluated in
// closed form here; the remainder is A(rho, z + z') + B(rho, z - z') from two
// sets of 2-D tables (256 log-spaced rho x 128), bilinear in (log rho, .).
#include <algorithm>
#include <cmath>
#include <complex>
#include <type_traits>

#include "dense.h"
#include "fill_dev.cuh"
#include "mgf.h"

namespace sldm {

// ---------------------------------------------------------------- complex FP64 helpers
struct cx {
  double r, i;
};
__host__ __device__ __forceinline__ cx mk(double r, double i = 0.0) { return {r, i}; }
__host__ __device__ __forceinline__ cx operator+(cx a, cx b) { return {a.r + b.r, a.i + b.i}; }
__host__ __device__ __forceinline__ cx operator-(cx a, cx b) { return {a.r - b.r, a.i - b.i}; }
__host__ __device__ __forceinline__ cx operator-(cx a) { return {-a.r, -a.i}; }
__host__ __device__ __forceinline__ cx operator*(cx a, cx b) { return {a.r * b.r - a.i * b.i, a.r * b.i + a.i * b.r}; }
__host__ __device__ __forceinline__ cx operator*(double s, cx a) { return {s * a.r, s * a.i}; }
__host__ __device__ __forceinline__ cx operator*(cx a, double s) { return {s * a.r, s * a.i}; }
__host__ __device__ __forceinline__ cx operator/(cx a, cx b) {
  const double d = b.r * b.r + b.i * b.i;
  return {(a.r * b.r + a.i * b.i) / d, (a.i * b.r - a.r * b.i) / d};
}
__device__ __forceinline__ cx cexp_(cx a) {
  double s, c;
  sincos(a.i, &s, &c);
  const double e = exp(a.r);
  return {e * c, e * s};
}
// exp(-j k R) for complex k: exp(Im k R) (cos(Re k R) - j sin(Re k R)); no exp when k is real
__device__ __forceinline__ cx eikr(cx k, double R) {
  double s, c;
  sincos(k.r * R, &s, &c);
  if (k.i == 0.0) return {c, -s};
  const double e = exp(k.i * R);
  return {e * c, -e * s};
}
// principal square root without cancellation: the larger of |Re|, |Im| comes
// from sqrt((|a| + |Re a|)/2), the other from Im a / (2 that)
__device__ __forceinline__ cx csqrt_(cx a) {
  if (a.r == 0.0 && a.i == 0.0) return {0.0, 0.0};
  const double t = sqrt(0.5 * (hypot(a.r, a.i) + fabs(a.r)));
  if (a.r >= 0.0) return {t, a.i / (2.0 * t)};
  return {fabs(a.i) / (2.0 * t), a.i < 0 ? -t : t};
}
// k_z = sqrt(k^2 - k_rho^2) with Im k_z <= 0
__device__ __forceinline__ cx kz_of(cx k, cx kr) {
  cx q = csqrt_(k * k - kr * kr);
  if (q.i > 0) q = -q;
  return q;
}

// J_n(z), n = 0, 1, complex z: periodic trapezoid rule of (1/2pi) int_0^2pi cos(n t - z sin t) dt
__device__ void bessel01_complex(cx z, cx* j0, cx* j1) {
  const double az = sqrt(z.r * z.r + z.i * z.i);
  const int M = 2 * (int(az) + 40);
  cx s0 = mk(0), s1 = mk(0);
  for (int m = 0; m < M; ++m) {
    double st, ct;
    sincospi(2.0 * m / M, &st, &ct);
    // cos(n t - z sin t) = (e^{i(nt - z st)} + e^{-i(nt - z st)})/2, z complex
    const cx ph = mk(z.r * st, z.i * st);  // z sin t
    // cos(w) for complex w = a + j b: cos a cosh b - j sin a sinh b
    auto ccos = [](cx w) {
      double sa, ca;
      sincos(w.r, &sa, &ca);
      if (w.i == 0.0) return cx{ca, 0.0};
      return cx{ca * cosh(w.i), -sa * sinh(w.i)};
    };
    s0 = s0 + ccos(-ph);
    // n = 1: cos(t - z sin t)
    const double t = 2.0 * M_PI * m / M;
    s1 = s1 + ccos(mk(t - ph.r, -ph.i));
  }
  *j0 = (1.0 / M) * s0;
  *j1 = (1.0 / M) * s1;
}

// ---------------------------------------------------------------- stack on the device
struct DevStack {
  int nl, l, pec, pad;
  double omega;
  cx eps[MGF_MAX_LAYERS];
  double mu[MGF_MAX_LAYERS];
  double d[MGF_MAX_LAYERS];  // thickness (finite layers)
  double zb, zu;             // bounds of layer l (+-1e300 for none)
  int top, bot;              // adjacent interfaces exist
};

constexpr double EPS0_ = 1.0 / (4e-7 * 3.14159265358979323846 * 299792458.0 * 299792458.0);
constexpr double MU0_ = 4e-7 * 3.14159265358979323846;
constexpr double C0_ = 299792458.0;

// generalised reflections (Gu, Gd) of line `te` (0 = e, 1 = h) seen from layer l
__device__ void reflections(const DevStack& S, cx kr, int te, cx* Gu, cx* Gd) {
  const double k0 = S.omega / C0_;
  cx Z[MGF_MAX_LAYERS], kz[MGF_MAX_LAYERS];
  for (int i = 0; i < S.nl; ++i) {
    // k_i = k0 sqrt(eps mu)
    cx k = csqrt_(S.mu[i] * S.eps[i]);
    k = k0 * k;
    kz[i] = kz_of(k, kr);
    Z[i] = te == 0 ? kz[i] / (S.omega * EPS0_ * S.eps[i]) : (S.omega * MU0_ * S.mu[i]) * (mk(1) / kz[i]);
  }
  auto fres = [&](int i, int j) { return (Z[j] - Z[i]) / (Z[j] + Z[i]); };
  cx up = mk(0);
  for (int i = 1; i <= S.l; ++i) {
    const cx f = fres(i, i - 1);
    if (i - 1 == 0) {
      up = f;
    } else {
      const cx ph = up * cexp_(mk(0, -2.0) * kz[i - 1] * mk(S.d[i - 1]));
      up = (f + ph) / (mk(1) + f * ph);
    }
  }
  const int last = S.nl - 1;
  cx down = S.pec ? mk(-1) : mk(0);
  for (int i = last - 1; i >= S.l; --i) {
    const cx f = fres(i, i + 1);
    if (i + 1 == last && !S.pec) {
      down = f;
    } else {
      const cx ph = down * cexp_(mk(0, -2.0) * kz[i + 1] * mk(S.d[i + 1]));
      down = (f + ph) / (mk(1) + f * ph);
    }
  }
  if (S.l == last) down = S.pec ? mk(-1) : mk(0);
  if (S.l == 0) up = mk(0);
  *Gu = up;
  *Gd = down;
}

// What the remainder's spectral kernels need at one node.  They are linear in the
// exponentials of the vertical argument: part 0 (argument s = z + z') single
// reflections minus the quasistatic images, in E1 = exp(-j k_z (2 zu - s)) and E2 =
// exp(-j k_z (s - 2 zb)), X1, X2 the static ones exp(-k_rho ..); part 1 (argument d = z - z')
// double reflections, in E3 = exp(-j k_z (2 dl + d)) and E4 = exp(-j k_z (2 dl - d)).  The
// reflections seen from layer l cost ~10^3 FP64 operations and depend on the node
// alone, so they are worked out once per node, not per (node, argument).
struct SpecNode {
  cx kz, kr;
  cx a[4], b[4];  // weight included: factors of E1 (E3) and E2 (E4) for xx, phi, zz, rho-z
  cx x1, x2;      // part 0: factors of X1 and X2 in rho-z
};
__device__ void spectral_node(const DevStack& S, const MgfStatic& Q, cx kr, cx f, int part, SpecNode& o) {
  const double k0 = S.omega / C0_;
  const cx epsl = S.eps[S.l];
  const double mur = S.mu[S.l];
  cx k = k0 * csqrt_(mur * epsl);
  const cx kz = kz_of(k, kr);
  const cx Ze = kz / (S.omega * EPS0_ * epsl);
  const cx Zh = (S.omega * MU0_ * mur) * (mk(1) / kz);
  cx Gue, Gde, Guh, Gdh;
  reflections(S, kr, 0, &Gue, &Gde);
  reflections(S, kr, 1, &Guh, &Gdh);
  const double dl = S.zu - S.zb;
  const cx zero = mk(0);
  const cx e2d = (S.top && S.bot) ? cexp_(mk(0, -2.0) * kz * mk(dl)) : zero;
  const cx De = mk(1) - Gue * Gde * e2d, Dh = mk(1) - Guh * Gdh * e2d;
  // reflected parts of the line functions at unit amplitude of each exponential
  auto Vi = [&](cx Z, cx g, cx D) { return (0.5 * Z) * (g / D); };
  auto Iv = [&](cx Z, cx g, cx D) { return (mk(0.5) / Z) * (g / D); };
  auto Ch = [&](cx g, cx D) { return 0.5 * (g / D); };
  const cx jw = mk(0, S.omega), kr2 = kr * kr;
  const cx cxx = mk(1) / (jw * mk(MU0_)), cph = EPS0_ * (jw / kr2);
  const cx czv = (mur * ((kr2 - kz * kz) / (EPS0_ * epsl * kr2))) / jw;
  const cx czh = ((S.omega * S.omega * MU0_ * mur * mur) * (mk(1) / kr2)) / jw;
  const cx crz = mk(0, mur) / kr;
  const cx gue = {Q.gue.r, Q.gue.i}, guh = {Q.guh.r, Q.guh.i}, gde = {Q.gde.r, Q.gde.i}, gdh = {Q.gdh.r, Q.gdh.i};
  o.kz = kz;
  o.kr = kr;
  o.x1 = o.x2 = zero;
  for (int side = 0; side < 2; ++side) {  // 0: E1 or E3, 1: E2 or E4
    // signs of the line functions: Vi (Gu, Gd, GuGd, GuGd), Iv (-Gu, -Gd, +, +), Vv (Gu, -Gd, GuGd, -GuGd)
    const cx ge = part == 0 ? (side == 0 ? Gue : Gde) : Gue * Gde;
    const cx gh = part == 0 ? (side == 0 ? Guh : Gdh) : Guh * Gdh;
    const double sIv = part == 0 ? -1.0 : 1.0, sVv = side == 0 ? 1.0 : -1.0;
    cx out[4];
    out[0] = Vi(Zh, gh, Dh) * cxx;
    out[1] = cph * (Vi(Ze, ge, De) - Vi(Zh, gh, Dh));
    out[2] = sIv * (czv * Iv(Ze, ge, De) + czh * Iv(Zh, gh, Dh));
    out[3] = sVv * (crz * (Ch(ge, De) - Ch(gh, Dh)));
    if (part == 0) {
      const cx g = mk(1) / (mk(0, 2) * kz);
      const cx se = side == 0 ? gue : gde, sh = side == 0 ? guh : gdh;
      out[0] = out[0] - (mur * sh) * g;
      out[1] = out[1] - (se * g) / epsl;
      out[2] = out[2] - (mur * (sh - 2.0 * se)) * g;
      // rho-z: the static single reflections exp(-k_rho zeta) (closed form in space)
      const cx c = f * ((mk(0, 0.5 * mur) / kr) * (se - sh));
      if (side == 0) o.x1 = -c;
      else o.x2 = c;
    }
    for (int c = 0; c < 4; ++c) (side == 0 ? o.a[c] : o.b[c]) = f * out[c];
  }
}

__global__ void mgf_nodes_kernel(DevStack S, MgfStatic Q, const double2* __restrict__ nodes, const double2* __restrict__ weights,
                                 int nnodes, int part, SpecNode* __restrict__ out) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= nnodes) return;
  const cx kr = {nodes[n].x, nodes[n].y};
  const cx f = (0.5 / 3.14159265358979323846) * (cx{weights[n].x, weights[n].y} * kr);
  SpecNode o;
  spectral_node(S, Q, kr, f, part, o);
  out[n] = o;
}
// exp(-x): no sine and cosine for a real exponent (the tail of a lossless stack)
__device__ __forceinline__ cx cexp_neg(cx x) {
  const double e = exp(-x.r);
  if (x.i == 0.0) return {e, 0.0};
  double s, c;
  sincos(x.i, &s, &c);
  return {e * c, -e * s};
}

// F[c][node][j] = w_node k_node g_c(k_node; arg_j) / (2 pi) for xx, phi, zz, rho-z; zero from
// the column group's last node on (group_end, see build_one)
constexpr int CT_J = 32;  // columns (arguments) of a group
__global__ void mgf_spectral_kernel(DevStack S, const SpecNode* __restrict__ sn, int nnodes, const double* __restrict__ args,
                                    int nargs, int part, const int* __restrict__ group_end, double2* F) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= int64_t(nnodes) * nargs) return;
  const int n = int(idx / nargs), j = int(idx % nargs);
  if (n >= group_end[j / CT_J]) return;  // not read either
  const SpecNode& o = sn[n];
  const double arg = args[j], dl = S.zu - S.zb;
  cx out[4] = {mk(0), mk(0), mk(0), mk(0)};
  auto add = [&](const cx* c, double zeta) {
    const cx E = cexp_neg(mk(0, 1) * o.kz * mk(zeta));
    for (int m = 0; m < 4; ++m) out[m] = out[m] + c[m] * E;
  };
  if (part == 0) {
    if (S.top) {
      add(o.a, 2 * S.zu - arg);
      out[3] = out[3] + o.x1 * cexp_neg(o.kr * mk(2 * S.zu - arg));
    }
    if (S.bot) {
      add(o.b, arg - 2 * S.zb);
      out[3] = out[3] + o.x2 * cexp_neg(o.kr * mk(arg - 2 * S.zb));
    }
  } else if (S.top && S.bot) {
    add(o.a, 2 * dl + arg);
    add(o.b, 2 * dl - arg);
  }
  for (int c = 0; c < 4; ++c) F[(int64_t(c) * nnodes + n) * nargs + j] = make_double2(out[c].r, out[c].i);
}

// J[order][i][n] = J_order(k_n rho_i): the real part for every node, the imaginary part
// Jc[order][i][n] for the ncomplex first nodes (the arc; the real-axis nodes have none)
__global__ void mgf_bessel_kernel(const double2* __restrict__ nodes, int nnodes, int ncomplex, const double* __restrict__ rho,
                                  int nr, double* __restrict__ J, double* __restrict__ Jc) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= int64_t(nnodes) * nr) return;
  const int i = int(idx / nnodes), n = int(idx % nnodes);
  const double2 k = nodes[n];
  if (n >= ncomplex) {
    // real axis (the tail panels, arguments up to ~1e4): the math library's J0, J1
    J[int64_t(i) * nnodes + n] = ::j0(k.x * rho[i]);
    J[int64_t(nr) * nnodes + int64_t(i) * nnodes + n] = ::j1(k.x * rho[i]);
    return;
  }
  // the elliptic arc (|z| below ~1e2): the periodic trapezoid rule is accurate to
  // rounding once it has 2(|z| + 40) points
  cx j0, j1;
  bessel01_complex(mk(k.x * rho[i], k.y * rho[i]), &j0, &j1);
  J[int64_t(i) * nnodes + n] = j0.r;
  J[int64_t(nr) * nnodes + int64_t(i) * nnodes + n] = j1.r;
  Jc[int64_t(i) * ncomplex + n] = j0.i;
  Jc[int64_t(nr) * ncomplex + int64_t(i) * ncomplex + n] = j1.i;
}

// part[split][c][i][j] = sum over the split's nodes n of J_{order(c)}[i][n] F[c][n][j].
// Rows i: rho, columns j: arguments; a CTA takes 32 rows (8 per warp) x 32 columns of
// one component, CT_N nodes of J staged in shared memory per step.  The FP64 pipe
// bounds it: two FMAs per real node and entry (J is real there), four on the arc
// (split 0); a column group ends where its exponentials have decayed (group_end).
// 5 x 5 cylinders on glass: 35.4 ms (complex J, five components, every node) -> 5.2 ms; the
// spectral values 12.3 -> 2 ms.
constexpr int CT_I = 8, CT_N = 32;
__global__ void __launch_bounds__(128) mgf_contract_kernel(const double* __restrict__ J, const double* __restrict__ Jc,
                                                           const double2* __restrict__ F, int nnodes, int ncomplex, int nr,
                                                           int nargs, int per_split, const int* __restrict__ group_end,
                                                           double2* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = blockIdx.x * CT_J + lane, i0 = blockIdx.y * (4 * CT_I);
  const int c = blockIdx.z % 4, split = blockIdx.z / 4;
  const int order = c == 3 ? 1 : 0;
  const double* Jo = J + int64_t(order) * nr * nnodes;
  const double* Jco = Jc + int64_t(order) * nr * ncomplex;
  const double2* Fc = F + int64_t(c) * nnodes * nargs;
  const int n_begin = split == 0 ? 0 : ncomplex + (split - 1) * per_split;
  const int n_end = min(group_end[blockIdx.x], split == 0 ? ncomplex : min(nnodes, n_begin + per_split));
  __shared__ double Js[4 * CT_I][CT_N];
  __shared__ double Ji[4 * CT_I][CT_N];
  double ar[CT_I], ai[CT_I];
#pragma unroll
  for (int ii = 0; ii < CT_I; ++ii) ar[ii] = ai[ii] = 0.0;
  // the arc apart: as a predicate in one loop its FMAs would take pipe slots on every node
  auto sum = [&](auto arc) {
    constexpr bool ARC = decltype(arc)::value;
    for (int n0 = n_begin; n0 < n_end; n0 += CT_N) {
      __syncthreads();
      for (int e = threadIdx.x; e < 4 * CT_I * CT_N; e += blockDim.x) {
        const int ii = e / CT_N, q = e % CT_N, gi = i0 + ii, gn = n0 + q;
        const bool ok = gi < nr && gn < n_end;
        Js[ii][q] = ok ? Jo[int64_t(gi) * nnodes + gn] : 0.0;
        if (ARC) Ji[ii][q] = ok ? Jco[int64_t(gi) * ncomplex + gn] : 0.0;
      }
      __syncthreads();
      if (j >= nargs) continue;
      const int nq = min(CT_N, n_end - n0);
#pragma unroll 2
      for (int q = 0; q < nq; ++q) {
        const double2 f = Fc[int64_t(n0 + q) * nargs + j];
#pragma unroll
        for (int ii = 0; ii < CT_I; ++ii) {
          const double a = Js[warp * CT_I + ii][q];
          ar[ii] = fma(a, f.x, ar[ii]);
          ai[ii] = fma(a, f.y, ai[ii]);
          if (ARC) {
            const double b = Ji[warp * CT_I + ii][q];
            ar[ii] = fma(-b, f.y, ar[ii]);
            ai[ii] = fma(b, f.x, ai[ii]);
          }
        }
      }
    }
  };
  if (split == 0) sum(std::true_type{});
  else sum(std::false_type{});
  if (j >= nargs) return;
  for (int ii = 0; ii < CT_I; ++ii) {
    const int i = i0 + warp * CT_I + ii;
    if (i < nr) part[((int64_t(split) * 4 + c) * nr + i) * nargs + j] = make_double2(ar[ii], ai[ii]);
  }
}

// table[c][i][j] = sum over splits of part (in split order), times -j for the order-1
// components; the z-rho component is -(rho-z) in part 0 and equal to it in part 1
__global__ void mgf_sum_splits(const double2* __restrict__ part, int nsplit, int64_t per, int nr, int nargs, int which,
                               double2* table) {
  const int64_t idx = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (idx >= per) return;
  double re = 0, im = 0;
  for (int sp = 0; sp < nsplit; ++sp) {
    const double2 v = part[int64_t(sp) * per + idx];
    re += v.x;
    im += v.y;
  }
  const int64_t plane = int64_t(nr) * nargs;
  const int c = int(idx / plane);
  if (c < 3) {
    table[idx] = make_double2(re, im);
    return;
  }
  table[idx + plane] = make_double2(im, -re);                                          // rho-z
  table[idx] = which == 0 ? make_double2(-im, re) : make_double2(im, -re);  // z-rho
}

// ---------------------------------------------------------------- host: nodes and tables
static void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
  x.resize(n);
  w.resize(n);
  for (int i = 0; i < n; ++i) {
    double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
    for (int it = 0; it < 100; ++it) {
      double p1 = 1.0, p2 = 0.0;
      for (int j = 1; j <= n; ++j) {
        const double p3 = p2;
        p2 = p1;
        p1 = ((2.0 * j - 1.0) * z * p2 - (j - 1.0) * p3) / j;
      }
      const double pp = n * (z * p1 - p2) / (z * z - 1.0);
      const double z1 = z;
      z = z1 - p1 / pp;
      if (std::fabs(z - z1) < 1e-16) {
        x[i] = -z;
        w[i] = 2.0 / ((1.0 - z * z) * pp * pp);
        break;
      }
      x[i] = -z;
      w[i] = 2.0 / ((1.0 - z * z) * pp * pp);
    }
  }
}

// Elliptic arc k(t) = a/2 (1 - cos t) + j b sin t over t in [0, pi] (n_e Gauss points),
// a = max(1.5 max Re k_i, 2 k0), b = min(a/2, 2/rho_max); then Gauss-Legendre panels
// (16 points) of width min(pi/rho_max, (k_end - a)/4) up to k_end = a + 32/zeta_min.
static void sommerfeld_nodes(const MgfStackHost& H, double omega, double rho_max, double zeta_min,
                             std::vector<double2>& nodes, std::vector<double2>& weights) {
  const double k0 = omega / C0_;
  double kmax = 0;
  for (size_t i = 0; i < H.eps.size(); ++i) kmax = std::max(kmax, std::abs((k0 * std::sqrt(H.eps[i] * H.mu[i])).real()));
  const double a = std::max(1.5 * kmax, 2.0 * k0);
  const double b = std::min(0.5 * a, 2.0 / rho_max);
  std::vector<double> x, w;
  gauss_legendre(MGF_N_ELLIPSE, x, w);
  nodes.clear();
  weights.clear();
  for (int i = 0; i < MGF_N_ELLIPSE; ++i) {
    const double t = 0.5 * M_PI * (x[i] + 1), wt = 0.5 * M_PI * w[i];
    nodes.push_back(make_double2(0.5 * a * (1 - std::cos(t)), b * std::sin(t)));
    weights.push_back(make_double2(0.5 * a * std::sin(t) * wt, b * std::cos(t) * wt));
  }
  const double kend = a + 32.0 / zeta_min;
  const double width = std::min(M_PI / rho_max, (kend - a) / 4);
  const int npan = int(std::ceil((kend - a) / width));
  gauss_legendre(MGF_PER_PANEL, x, w);
  for (int p = 0; p < npan; ++p) {
    const double mid = a + width * (p + 0.5);
    for (int q = 0; q < MGF_PER_PANEL; ++q) {
      nodes.push_back(make_double2(mid + 0.5 * width * x[q], 0.0));
      weights.push_back(make_double2(0.5 * width * w[q], 0.0));
    }
  }
}

static DevStack dev_stack(const MgfStackHost& H, double omega) {
  DevStack S{};
  S.nl = int(H.eps.size());
  S.l = H.l;
  S.pec = H.pec;
  S.omega = omega;
  for (int i = 0; i < S.nl; ++i) {
    S.eps[i] = {H.eps[i].real(), H.eps[i].imag()};
    S.mu[i] = H.mu[i];
    S.d[i] = H.d[i];
  }
  S.zb = H.zb;
  S.zu = H.zu;
  S.top = H.top;
  S.bot = H.bot;
  return S;
}

static void build_one(const MgfStackHost& H, const MgfStatic& Q, double omega, const std::vector<double>& rho,
                      const std::vector<double>& args, int part, double zeta_min, double2* out, cudaStream_t s) {
  std::vector<double2> nodes, weights;
  sommerfeld_nodes(H, omega, rho.back() / 1.0, zeta_min, nodes, weights);
  const int nn = int(nodes.size()), nr = int(rho.size()), na = int(args.size());
  const int ncomplex = std::min(MGF_N_ELLIPSE, nn);
  // A column's exponentials fall at least like exp(-kappa zeta), kappa = sqrt(k_rho^2 -
  // Re k_l^2) on the real axis, zeta its smallest distance to an image: past kappa zeta =
  // 60 (1e-26; the other factors grow like a power of k_rho) nothing reaches the sum's
  // rounding, and the group of 32 columns ends there.
  const double k0 = omega / C0_, kl2 = std::real(k0 * k0 * H.eps[H.l] * H.mu[H.l]);
  std::vector<int> gend;
  for (int j0 = 0; j0 < na; j0 += CT_J) {
    double zeta = 1e300;
    for (int j = j0; j < std::min(na, j0 + CT_J); ++j) {
      if (part == 0 && H.top) zeta = std::min(zeta, 2 * H.zu - args[j]);
      if (part == 0 && H.bot) zeta = std::min(zeta, args[j] - 2 * H.zb);
      if (part == 1) zeta = std::min(zeta, 2 * (H.zu - H.zb) - args[j]);
    }
    int e = nn;
    if (zeta > 0) {
      const double kap = 60.0 / zeta, kmax = std::sqrt(std::max(0.0, kl2 + kap * kap));
      e = ncomplex;
      while (e < nn && nodes[e].x <= kmax) ++e;
    }
    gend.push_back(e);
  }
  DBuf<double2> dn, dw, F;
  DBuf<double> dr, da, J, Jc;
  DBuf<int> dg;
  DBuf<SpecNode> sn;
  dn.upload(nodes, s);
  dw.upload(weights, s);
  dr.upload(rho, s);
  da.upload(args, s);
  dg.upload(gend, s);
  F.alloc(size_t(nn) * na * 4);
  J.alloc(size_t(2) * nr * nn);
  Jc.alloc(size_t(2) * nr * ncomplex);
  sn.alloc(nn);
  const DevStack S = dev_stack(H, omega);
  {
    ScopedTimer tm("mgf_tables", s);
    mgf_nodes_kernel<<<unsigned((nn + 63) / 64), 64, 0, s>>>(S, Q, dn.p, dw.p, nn, part, sn.p), ::sldm::count_launch();
    const int64_t tot = int64_t(nn) * na;
    mgf_spectral_kernel<<<unsigned((tot + 127) / 128), 128, 0, s>>>(S, sn.p, nn, da.p, na, part, dg.p, F.p),
        ::sldm::count_launch();
    const int64_t totb = int64_t(nn) * nr;
    mgf_bessel_kernel<<<unsigned((totb + 127) / 128), 128, 0, s>>>(dn.p, nn, ncomplex, dr.p, nr, J.p, Jc.p),
        ::sldm::count_launch();
    // split the real-axis nodes so that the product runs ~16 CTAs per SM (short ones included)
    const int base = ((na + CT_J - 1) / CT_J) * ((nr + 4 * CT_I - 1) / (4 * CT_I)) * 4;
    const int want = std::max(1, std::min(63, (16 * 152 + base - 1) / base));
    const int per_split = std::max(CT_N, ((nn - ncomplex + want - 1) / want + CT_N - 1) / CT_N * CT_N);
    const int nsplit = 1 + (nn - ncomplex + per_split - 1) / per_split;
    const int64_t per = int64_t(4) * nr * na;
    DBuf<double2> sums;
    sums.alloc(size_t(nsplit) * per);
    mgf_contract_kernel<<<dim3((na + CT_J - 1) / CT_J, (nr + 4 * CT_I - 1) / (4 * CT_I), 4 * nsplit), 128, 0, s>>>(
        J.p, Jc.p, F.p, nn, ncomplex, nr, na, per_split, dg.p, sums.p),
        ::sldm::count_launch();
    mgf_sum_splits<<<unsigned((per + 255) / 256), 256, 0, s>>>(sums.p, nsplit, per, nr, na, part, out), ::sldm::count_launch();
    SLDM_CUDA(cudaStreamSynchronize(s));
  }
  SLDM_CUDA(cudaGetLastError());
  SLDM_CUDA(cudaStreamSynchronize(s));
}

void mgf_build_tables(const MgfStackHost& H, double omega, double rho_min, double rho_max, double zmin, double zmax,
                      MgfTables& T, cudaStream_t s) {
  T.nr = MGF_NR;
  T.ns = MGF_NS;
  T.nd = MGF_ND;
  std::vector<double> rho(T.nr), sv(T.ns), dv(T.nd);
  for (int i = 0; i < T.nr; ++i)
    rho[i] = std::exp(std::log(rho_min) + (std::log(rho_max) - std::log(rho_min)) * i / (T.nr - 1));
  for (int j = 0; j < T.ns; ++j) sv[j] = 2 * zmin + (2 * zmax - 2 * zmin) * j / (T.ns - 1);
  for (int j = 0; j < T.nd; ++j) dv[j] = (zmax - zmin) * j / (T.nd - 1);
  T.lr0 = std::log(rho_min);
  T.lr1 = std::log(rho_max);
  T.s0 = 2 * zmin;
  T.s1 = 2 * zmax;
  T.d1 = zmax - zmin;
  T.A.alloc(size_t(5) * T.nr * T.ns);
  T.B.alloc(size_t(5) * T.nr * T.nd);
  // Objects may rest on an interface, where z + z' - 2 z_b = 0 and nothing decays
  // exponentially: the Sommerfeld tail is cut where exp(-k_rho zeta_floor) < 1e-14,
  // zeta_floor = 1/16 of the objects' height (the remainder decays algebraically
  // once every static image is out).
  const double zfloor = zmax > zmin ? (zmax - zmin) / 16 : 1e-3 * rho_max;
  double zeta_a = 1.0;
  {
    bool any = false;
    double zm = 1e300;
    if (H.top) {
      zm = std::min(zm, 2 * H.zu - 2 * zmax);
      any = true;
    }
    if (H.bot) {
      zm = std::min(zm, 2 * zmin - 2 * H.zb);
      any = true;
    }
    if (any) zeta_a = std::max(zm, zfloor);
  }
  build_one(H, T.Q, omega, rho, sv, 0, zeta_a, T.A.p, s);
  T.hasB = H.top && H.bot;
  if (H.top && H.bot) {
    const double zeta_b = std::max(2 * (H.zu - H.zb) - (zmax - zmin), zfloor);
    build_one(H, T.Q, omega, rho, dv, 1, zeta_b, T.B.p, s);
  } else {
    T.B.zero(s);
  }
}

// ---------------------------------------------------------------- reflected fill of L^A_m, L^phi_m
// The tables as bilinear cells: cell (i, j) holds, for the four components the fill
// needs (xx, phi, zz, rho-z: the z-rho component is -(rho-z) in A and equal to it in
// B), a = f_00, b = f_10 - f_00, c = f_01 - f_00, d = f_11 - f_10 - f_01 + f_00, so a
// value costs three FMAs per real part and its 16 operands are 256 contiguous bytes.
constexpr int CELL_C = 4;
__global__ void mgf_cells_kernel(const double2* __restrict__ t, int nr, int ny, double2* __restrict__ cells) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (nr - 1) * ny * CELL_C) return;
  const int comp = idx % CELL_C, ij = idx / CELL_C, i = ij / ny, j = ij % ny, j1 = min(j + 1, ny - 1);
  const double2* f = t + int64_t(comp == 3 ? 4 : comp) * nr * ny;
  const double2 f00 = f[int64_t(i) * ny + j], f10 = f[int64_t(i + 1) * ny + j], f01 = f[int64_t(i) * ny + j1],
                f11 = f[int64_t(i + 1) * ny + j1];
  double2* o = cells + int64_t(idx) * 4;
  o[0] = f00;
  o[1] = make_double2(f10.x - f00.x, f10.y - f00.y);
  o[2] = make_double2(f01.x - f00.x, f01.y - f00.y);
  o[3] = make_double2((f11.x - f10.x) - (f01.x - f00.x), (f11.y - f10.y) - (f01.y - f00.y));
}

// Cell index and offset of a fractional index f in [0, n - 1] (clamped there):
// round f - 1/2 by adding and subtracting 1.5 2^52, no conversion on the FP64 pipe.
__device__ __forceinline__ int cell_of(double f, int last, double& t) {
  if (__double2hiint(f) < 0) f = 0.0;
  const double h = f - 0.5, m = __dadd_rn(h, 6755399441055744.0);
  int i = __double2loint(m);
  t = f - __dsub_rn(m, 6755399441055744.0);
  if (i > last) {  // the table's edge, up to rounding
    i = last;
    t = 1.0;
  }
  return i;
}
__device__ __forceinline__ cx cell_value(const double2* __restrict__ c, double tx, double ty) {
  const double2 a = c[0], b = c[1], g = c[2], d = c[3];
  return {fma(tx, fma(ty, d.x, b.x), fma(ty, g.x, a.x)), fma(tx, fma(ty, d.y, b.y), fma(ty, g.y, a.y))};
}

// What the fill needs of the stack, worked out on the host.
struct ReflArgs {
  cx k;                        // of the objects' layer
  double ys, ye;               // k.r, k.i in steps of the wave tables
  double zu2, zb2;             // 2 zu, 2 zb
  double kxx_u, kxx_d;         // image coefficients: xx mu_r g_h, phi g_e / eps_r, zz mu_r (g_h - 2 g_e)
  cx kph_u, kph_d, kzz_u, kzz_d;
  cx kzr_u, kzr_d;             // mu_r (g_e - g_h) of the static rho-z images
  const double2 *ca, *cb;      // cells of the two tables
  int nr, ns, nd;
  double fx1, fx0;             // cell index of rho: fx1 log2(rho^2) + fx0
  double s0, ss, sd;           // (z + z' - s0) ss, |z - z'| sd
  double rmin2, inv_rmin;
};


// Pair (t, s) touches through an interface when the triangles share a vertex on
// it: bits 0-2 (bottom) and 4-6 (top) of onmask flag vertices on the interfaces.
__device__ __forceinline__ bool touch_through(const int32_t* tri, int t, int s, int mt, int ms, int shift) {
  if (!((mt >> shift) & 7) || !((ms >> shift) & 7)) return false;
  for (int i = 0; i < 3; ++i) {
    if (!((mt >> (shift + i)) & 1)) continue;
    for (int j = 0; j < 3; ++j)
      if (((ms >> (shift + j)) & 1) && tri[3 * t + i] == tri[3 * s + j]) return true;
  }
  return false;
}

// acc += s b for a real s
__device__ __forceinline__ void fmac(cx& acc, double s, cx b) {
  acc.r = fma(s, b.r, acc.r);
  acc.i = fma(s, b.i, acc.i);
}
// acc += a b
__device__ __forceinline__ void cmac(cx& acc, cx a, cx b) {
  acc.r = fma(-a.i, b.i, fma(a.r, b.r, acc.r));
  acc.i = fma(a.i, b.r, fma(a.r, b.i, acc.i));
}

// One thread per (test, source) triangle pair of a block task, 6 x 6 points: the
// images (spherical waves and static z-rho / rho-z) and the tabulated remainder.
// An interface's images are left out for pairs touching through it (they are
// integrated apart by fill_reflected_touch); a coincident image point adds 0.
// The dyadic kernel (xx, zz, and with rhohat = (hx, hy) the vectors R = grz rhohat, Z =
// gzr rhohat) meets f_i(r) = s_i (r - V_i) / (2 A) and f'_j alike, so the sums over
// source points of kernel x (1, r') and then over test points of those x (1, r) give
// the 3x3 block at the end of the pair.  A task of one triangle set against itself is
// symmetric (gzr(r, r') = -grz(r', r) in the images and the A table, and with the sign of
// z - z' in the B table): pairs s >= t, scattered to both places.
// Bound by the FP64 pipe.  5 x 5 cylinders on glass (one interface): 95 ms (every pair,
// ~300 operations per evaluation, the dyadic products and 3x3 block per test point) -> 48 ms
// with half the pairs -> 26 ms; 2,048-triangle wire between two interfaces: 119 -> 38 ms.
template <class C, bool TOP, bool BOT>
__global__ void __launch_bounds__(128, 2) fill_reflected_kernel(const RTask* __restrict__ tasks, const double* __restrict__ geo,
                                                                const int32_t* __restrict__ tri_edge,
                                                                const int32_t* __restrict__ tri,
                                                                const int32_t* __restrict__ onmask, const ReflArgs P, C* LA,
                                                                int64_t ldA, C* LP, int64_t ldP) {
  constexpr bool HASB = TOP && BOT;
  __shared__ WaveTab wt;
  __shared__ LogTab lt;
  const RTask tk = tasks[blockIdx.y];
  const int64_t total = int64_t(tk.ntest) * tk.nsrc;
  if (int64_t(blockIdx.x) * blockDim.x >= total) return;
  wave_tab_fill(wt, P.k.i != 0.0);
  log_tab_fill(lt);
  __syncthreads();
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= total) return;
  const int t = tk.t0 + int(p / tk.nsrc), sidx = tk.s0 + int(p % tk.nsrc);
  const bool sym = tk.t0 == tk.s0 && tk.ntest == tk.nsrc;
  if (sym && sidx < t) return;
  const double* gt = geo + size_t(t) * GEO_STRIDE;
  const double* gs = geo + size_t(sidx) * GEO_STRIDE;
  const bool lossy = P.k.i != 0.0;
  const int mt = onmask[t], ms = onmask[sidx];
  const double img_b = touch_through(tri, t, sidx, mt, ms, 0) ? 0.0 : INV4PI;
  const double img_t = touch_through(tri, t, sidx, mt, ms, 4) ? 0.0 : INV4PI;
  const double dcx = gt[GEO_C] - gs[GEO_C], dcy = gt[GEO_C + 1] - gs[GEO_C + 1];
  const cx zero = mk(0);
  cx xS = zero, xMx = zero, xMy = zero, xRx = zero, xRy = zero, x0 = zero;  // xx: r.r', r', r, 1
  cx zS = zero, zM = zero, zR = zero, z0 = zero;                            // zz: z z', z', z, 1
  cx rS = zero, rMx = zero, rMy = zero, rR = zero, r0x = zero, r0y = zero;  // R: r.R z', R z', r.R, R
  cx cS = zero, cM = zero, cRx = zero, cRy = zero, c0x = zero, c0y = zero;  // Z: z Z.r', Z.r', z Z, Z
  cx lp = zero;
#pragma unroll 1
  for (int q = 0; q < 6; ++q) {
    const double tx = gt[GEO_RHO + 3 * q], ty = gt[GEO_RHO + 3 * q + 1], tz = gt[GEO_RHO + 3 * q + 2];
    const double zz = gt[GEO_C + 2] + tz;
    cx a0 = zero, ax = zero, ay = zero, az0 = zero, azz = zero, bx = zero, by = zero, bxz = zero, byz = zero;
    cx dx0 = zero, dy0 = zero, dr = zero, sphi = zero;
#pragma unroll 1
    for (int sq = 0; sq < 6; ++sq) {
      const double px = gs[GEO_RHO + 3 * sq], py = gs[GEO_RHO + 3 * sq + 1], pz = gs[GEO_RHO + 3 * sq + 2];
      const double w = gs[GEO_W + sq];
      const double zp = gs[GEO_C + 2] + pz;
      const double dx = dcx + (tx - px), dy = dcy + (ty - py);
      const double rho2 = fma(dx, dx, dy * dy);
      const double irho = rho2 > 0 ? rsqrt_pos(rho2) : 0.0;
      const double rho = rho2 * irho;
      const double zs = zz + zp;
      cx gxx = zero, gphi = zero, gzz = zero, grz = zero;
      // quasistatic images: spherical waves exp(-j k R)/(4 pi R) and the static
      // rho-z image rho / (4 pi R (R + zeta)) from the image points
      auto image = [&](double zeta, double img, double kxx, cx kph, cx kzz, cx krz) {
        const double R2 = fma(zeta, zeta, rho2);
        if (!(R2 > 0)) return;
        const double r1 = rsqrt_pos(R2), R = R2 * r1, iR = img * r1;
        double c, sn;
        wave_cis(wt, P.ys * R, c, sn);
        const double am = lossy ? iR * wave_exp2(wt, P.ye * R) : iR;
        const cx G = {am * c, -am * sn};
        const double F = iR * rho * recip_pos(R + zeta);
        fmac(gxx, kxx, G);
        cmac(gphi, kph, G);
        cmac(gzz, kzz, G);
        fmac(grz, F, krz);
      };
      if (TOP) image(P.zu2 - zs, img_t, P.kxx_u, P.kph_u, P.kzz_u, P.kzr_u);
      if (BOT) image(zs - P.zb2, img_b, P.kxx_d, P.kph_d, P.kzz_d, -P.kzr_d);
      // tabulated remainder (one bilinear cell for the components of a table)
      const double rc2 = __double_as_longlong(rho2) > __double_as_longlong(P.rmin2) ? rho2 : P.rmin2;
      double fx, fy;
      const int ix = cell_of(fma(P.fx1, log2_pos(lt, rc2), P.fx0), P.nr - 2, fx);
      const int iy = cell_of((zs - P.s0) * P.ss, P.ns - 2, fy);
      const double2* ca = P.ca + (int64_t(ix) * P.ns + iy) * (4 * CELL_C);
      gxx = gxx + cell_value(ca, fx, fy);
      gphi = gphi + cell_value(ca + 4, fx, fy);
      gzz = gzz + cell_value(ca + 8, fx, fy);
      // the S1 (z-rho, rho-z) remainders vanish linearly at rho = 0: below rho_min scale by rho / rho_min
      const double lin = rc2 == rho2 ? 1.0 : rho * P.inv_rmin;
      fmac(grz, lin, cell_value(ca + 12, fx, fy));
      cx gzr = -grz;
      if (HASB) {
        const double dd = zz - zp;
        const int iyb = cell_of(fabs(dd) * P.sd, P.nd - 2, fy);
        const double2* cb = P.cb + (int64_t(ix) * P.nd + iyb) * (4 * CELL_C);
        gxx = gxx + cell_value(cb, fx, fy);
        gphi = gphi + cell_value(cb + 4, fx, fy);
        gzz = gzz + cell_value(cb + 8, fx, fy);
        const double ls = dd > 0 ? lin : (dd < 0 ? -lin : 0.0);
        const cx b = cell_value(cb + 12, fx, fy);
        fmac(grz, ls, b);
        fmac(gzr, ls, b);
      }
      const double whx = w * (dx * irho), why = w * (dy * irho);
      const cx wxx = w * gxx, wzz = w * gzz;
      a0 = a0 + wxx;
      fmac(ax, px, wxx);
      fmac(ay, py, wxx);
      az0 = az0 + wzz;
      fmac(azz, pz, wzz);
      fmac(sphi, w, gphi);
      const cx wrx = whx * grz, wry = why * grz;
      bx = bx + wrx;
      by = by + wry;
      fmac(bxz, pz, wrx);
      fmac(byz, pz, wry);
      if (HASB) {
        const cx wzx = whx * gzr, wzy = why * gzr;
        dx0 = dx0 + wzx;
        dy0 = dy0 + wzy;
        fmac(dr, px, wzx);
        fmac(dr, py, wzy);
      } else {  // gzr = -grz
        fmac(dr, -px, wrx);
        fmac(dr, -py, wry);
      }
    }
    if (!HASB) {
      dx0 = -bx;
      dy0 = -by;
    }
    const double wq = gt[GEO_W + q], wx = wq * tx, wy = wq * ty, wz = wq * tz;
    fmac(xS, wx, ax);
    fmac(xS, wy, ay);
    fmac(xMx, wq, ax);
    fmac(xMy, wq, ay);
    fmac(xRx, wx, a0);
    fmac(xRy, wy, a0);
    fmac(x0, wq, a0);
    fmac(zS, wz, azz);
    fmac(zM, wq, azz);
    fmac(zR, wz, az0);
    fmac(z0, wq, az0);
    fmac(rS, wx, bxz);
    fmac(rS, wy, byz);
    fmac(rMx, wq, bxz);
    fmac(rMy, wq, byz);
    fmac(rR, wx, bx);
    fmac(rR, wy, by);
    fmac(r0x, wq, bx);
    fmac(r0y, wq, by);
    fmac(cS, wz, dr);
    fmac(cM, wq, dr);
    fmac(cRx, wz, dx0);
    fmac(cRy, wz, dy0);
    fmac(c0x, wq, dx0);
    fmac(c0y, wq, dy0);
    fmac(lp, wq, sphi);
  }
  // (r + a_i).T.(r' + b_j) from the sums (a = c - V, GEO_AV)
  const cx base = (xS + zS) + (rS + cS);
  for (int i = 0; i < 3; ++i) {
    const double ax = gt[GEO_AV + 3 * i], ay = gt[GEO_AV + 3 * i + 1], az = gt[GEO_AV + 3 * i + 2];
    cx bi = base;  // terms without b_j
    fmac(bi, ax, xMx + rMx);
    fmac(bi, ay, xMy + rMy);
    fmac(bi, az, zM + cM);
    for (int j = 0; j < 3; ++j) {
      const double ux = gs[GEO_AV + 3 * j], uy = gs[GEO_AV + 3 * j + 1], uz = gs[GEO_AV + 3 * j + 2];
      cx v = bi;
      fmac(v, ux, xRx + cRx);
      fmac(v, uy, xRy + cRy);
      fmac(v, uz, zR + rR);
      fmac(v, fma(ax, ux, ay * uy), x0);
      fmac(v, az * uz, z0);
      fmac(v, ax * uz, r0x);
      fmac(v, ay * uz, r0y);
      fmac(v, az * ux, c0x);
      fmac(v, az * uy, c0y);
      v = (gt[GEO_SIG + i] * gs[GEO_SIG + j]) * v;
      const int64_t row = tri_edge[3 * t + i], col = tri_edge[3 * sidx + j];
      M<decltype(LA->x)>::add(LA, row * ldA + col, v.r, v.i);
      if (sym && sidx != t) M<decltype(LA->x)>::add(LA, col * ldA + row, v.r, v.i);
    }
  }
  const double sc = 1.0 / (gt[GEO_A] * gs[GEO_A]);
  auto addp = [&](C* dp) {
    dp->x = decltype(dp->x)(double(dp->x) + sc * lp.r);
    dp->y = decltype(dp->y)(double(dp->y) + sc * lp.i);
  };
  addp(LP + int64_t(t) * ldP + sidx);
  if (sym && sidx != t) addp(LP + int64_t(sidx) * ldP + t);
}

// ---------------------------------------------------------------- pairs touching through an interface
// Gauss-Legendre nodes and weights on [0, 1] of the Duffy rule
static __constant__ double c_duffy_x[MGF_DUFFY_N], c_duffy_w[MGF_DUFFY_N];

// The point of triangle (a, b, c) nearest to r: the projection on the plane when
// inside, else the nearest point of the three edges.
__device__ void closest_point(const double* r, const double* a, const double* b, const double* c, double* out) {
  double v0[3], v1[3], n[3];
  for (int d = 0; d < 3; ++d) {
    v0[d] = b[d] - a[d];
    v1[d] = c[d] - a[d];
  }
  n[0] = v0[1] * v1[2] - v0[2] * v1[1];
  n[1] = v0[2] * v1[0] - v0[0] * v1[2];
  n[2] = v0[0] * v1[1] - v0[1] * v1[0];
  const double nn = n[0] * n[0] + n[1] * n[1] + n[2] * n[2];
  const double h = ((r[0] - a[0]) * n[0] + (r[1] - a[1]) * n[1] + (r[2] - a[2]) * n[2]) / nn;
  double p[3], v2[3];
  for (int d = 0; d < 3; ++d) {
    p[d] = r[d] - h * n[d];
    v2[d] = p[d] - a[d];
  }
  const double d00 = v0[0] * v0[0] + v0[1] * v0[1] + v0[2] * v0[2];
  const double d01 = v0[0] * v1[0] + v0[1] * v1[1] + v0[2] * v1[2];
  const double d11 = v1[0] * v1[0] + v1[1] * v1[1] + v1[2] * v1[2];
  const double d20 = v2[0] * v0[0] + v2[1] * v0[1] + v2[2] * v0[2];
  const double d21 = v2[0] * v1[0] + v2[1] * v1[1] + v2[2] * v1[2];
  const double den = d00 * d11 - d01 * d01;
  const double bv = (d11 * d20 - d01 * d21) / den, bw = (d00 * d21 - d01 * d20) / den;
  if (bv >= 0 && bw >= 0 && bv + bw <= 1) {
    for (int d = 0; d < 3; ++d) out[d] = p[d];
    return;
  }
  const double* E[4] = {a, b, c, a};
  double best = 1e300;
  for (int e = 0; e < 3; ++e) {
    const double* u = E[e];
    const double* v = E[e + 1];
    double uv[3], ur[3];
    for (int d = 0; d < 3; ++d) {
      uv[d] = v[d] - u[d];
      ur[d] = r[d] - u[d];
    }
    double t = (ur[0] * uv[0] + ur[1] * uv[1] + ur[2] * uv[2]) / (uv[0] * uv[0] + uv[1] * uv[1] + uv[2] * uv[2]);
    t = fmin(fmax(t, 0.0), 1.0);
    double qd[3], dist = 0;
    for (int d = 0; d < 3; ++d) {
      qd[d] = u[d] + t * uv[d];
      dist += (r[d] - qd[d]) * (r[d] - qd[d]);
    }
    dist = sqrt(dist);
    if (dist < best) {
      best = dist;
      for (int d = 0; d < 3; ++d) out[d] = qd[d];
    }
  }
}

// One group of 8 threads per pair touching through an interface (thread q < 6:
// outer point q of the test triangle): that interface's images over the mirrored
// source triangle (x', y', 2 z_I - z'), where the RWG keeps its transverse part and
// flips its z part.  xx, phi, zz: the spherical wave with 1/R and R in closed form
// over the mirrored triangle and the rest by its 6 points; z-rho, rho-z: the static
// kernel (r - r'')_t / (4 pi R (R + zeta)) by the Duffy rule (n x n Gauss points on
// each of the three parts of the mirrored triangle split at its point nearest r).
template <class C>
__global__ void fill_reflected_touch(const int32_t* __restrict__ pairs, int npairs, const double* __restrict__ geo,
                                     const double* __restrict__ xyz, const int32_t* __restrict__ tri,
                                     const int32_t* __restrict__ tri_edge, DevStack S, MgfStatic Q, C* LA, int64_t ldA, C* LP,
                                     int64_t ldP) {
  const int64_t gt_ = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int p = int(gt_ >> 3), q = int(gt_ & 7);
  const bool valid = p < npairs;
  const int t = valid ? pairs[3 * p] : 0, sidx = valid ? pairs[3 * p + 1] : 0, top = valid ? pairs[3 * p + 2] : 0;
  const bool act = valid && q < 6;
  double m[20];
#pragma unroll
  for (int i = 0; i < 20; ++i) m[i] = 0.0;
  const double* gt = geo + size_t(t) * GEO_STRIDE;
  const double* gs = geo + size_t(sidx) * GEO_STRIDE;
  if (act) {
    const double k0 = S.omega / C0_;
    const cx epsl = S.eps[S.l];
    const double mur = S.mu[S.l];
    const cx k = k0 * csqrt_(mur * epsl);
    const cx k2 = k * k;
    const double zI = top ? S.zu : S.zb;
    const cx ge = top ? cx{Q.gue.r, Q.gue.i} : cx{Q.gde.r, Q.gde.i};
    const cx gh = top ? cx{Q.guh.r, Q.guh.i} : cx{Q.gdh.r, Q.gdh.i};
    const cx czr = top ? -(mur * (ge - gh)) : mur * (ge - gh), crz = -czr;
    const cx cxx = mur * gh, czz = mur * (gh - 2.0 * ge), cphi = ge / epsl;
    double Bm[3][3];  // mirrored source vertices
    for (int j = 0; j < 3; ++j)
      for (int d = 0; d < 3; ++d) Bm[j][d] = d == 2 ? 2 * zI - xyz[3 * tri[3 * sidx + j] + 2] : xyz[3 * tri[3 * sidx + j] + d];
    double r[3], f[3][3];
    for (int d = 0; d < 3; ++d) r[d] = gt[GEO_C + d] + gt[GEO_RHO + 3 * q + d];
    for (int i = 0; i < 3; ++i)
      for (int d = 0; d < 3; ++d) f[i][d] = gt[GEO_SIG + i] * (gt[GEO_RHO + 3 * q + d] + gt[GEO_AV + 3 * i + d]);
    // int G and int p G over the mirrored triangle
    cx I0 = mk(0), Ip[3] = {mk(0), mk(0), mk(0)};
    for (int j = 0; j < 6; ++j) {
      double rs[3];
      for (int d = 0; d < 3; ++d) rs[d] = gs[GEO_C + d] + gs[GEO_RHO + 3 * j + d];
      rs[2] = 2 * zI - rs[2];
      const double dx = r[0] - rs[0], dy = r[1] - rs[1], dz = r[2] - rs[2];
      const cd g = green_smooth(cd{k.r, k.i}, sqrt(dx * dx + dy * dy + dz * dz));
      const double w = gs[GEO_W + j];
      I0 = I0 + w * cx{g.r, g.i};
      for (int d = 0; d < 3; ++d) Ip[d] = Ip[d] + (w * rs[d]) * cx{g.r, g.i};
    }
    Pot P;
    potentials(r, Bm[0], Bm[1], Bm[2], P);
    I0 = I0 + mk(INV4PI * P.inv_r) - (0.5 * INV4PI * P.r) * k2;
    for (int d = 0; d < 3; ++d)
      Ip[d] = Ip[d] + mk(INV4PI * (P.por[d] + P.rho[d] * P.inv_r)) - (0.5 * INV4PI * (P.pr[d] + P.rho[d] * P.r)) * k2;
    // static z-rho kernel by the Duffy rule: J0 = int W, J1[d][e] = int W_d p_e
    double J0[2] = {0, 0}, J1[2][3] = {{0, 0, 0}, {0, 0, 0}};
    {
      double Qp[3];
      closest_point(r, Bm[0], Bm[1], Bm[2], Qp);
      double e1[3], e2[3];
      for (int d = 0; d < 3; ++d) {
        e1[d] = Bm[1][d] - Bm[0][d];
        e2[d] = Bm[2][d] - Bm[0][d];
      }
      const double fx_ = e1[1] * e2[2] - e1[2] * e2[1], fy_ = e1[2] * e2[0] - e1[0] * e2[2], fz_ = e1[0] * e2[1] - e1[1] * e2[0];
      const double full = sqrt(fx_ * fx_ + fy_ * fy_ + fz_ * fz_);
      for (int sub = 0; sub < 3; ++sub) {
        const double* P1 = Bm[sub];
        const double* P2 = Bm[(sub + 1) % 3];
        double a1[3], a2v[3];
        for (int d = 0; d < 3; ++d) {
          a1[d] = P1[d] - Qp[d];
          a2v[d] = P2[d] - P1[d];
        }
        const double cx_ = a1[1] * a2v[2] - a1[2] * a2v[1], cy_ = a1[2] * a2v[0] - a1[0] * a2v[2],
                     cz_ = a1[0] * a2v[1] - a1[1] * a2v[0];
        const double a2 = sqrt(cx_ * cx_ + cy_ * cy_ + cz_ * cz_);
        if (a2 <= 1e-12 * full) continue;
        for (int iu = 0; iu < MGF_DUFFY_N; ++iu) {
          const double u = c_duffy_x[iu];
          for (int iv = 0; iv < MGF_DUFFY_N; ++iv) {
            const double v = c_duffy_x[iv];
            const double wt = a2 * u * c_duffy_w[iu] * c_duffy_w[iv];
            double pt[3];
            for (int d = 0; d < 3; ++d) pt[d] = Qp[d] + u * a1[d] + u * v * a2v[d];
            const double dx = r[0] - pt[0], dy = r[1] - pt[1], dz = r[2] - pt[2];
            const double R = sqrt(dx * dx + dy * dy + dz * dz);
            const double den = R * (R + fabs(dz));
            if (!(den > 0)) continue;
            const double s_ = wt * INV4PI / den;
            const double wx = s_ * dx, wy = s_ * dy;
            J0[0] += wx;
            J0[1] += wy;
            for (int e = 0; e < 3; ++e) {
              J1[0][e] += wx * pt[e];
              J1[1][e] += wy * pt[e];
            }
          }
        }
      }
    }
    const double wq = gt[GEO_W + q];
    for (int j = 0; j < 3; ++j) {
      const double sb = gs[GEO_SIG + j];
      cx in[3];
      for (int d = 0; d < 3; ++d) in[d] = Ip[d] - Bm[j][d] * I0;  // int (p'' - v''_j) G
      const double tj = (J1[0][0] - Bm[j][0] * J0[0]) + (J1[1][1] - Bm[j][1] * J0[1]);
      const double zj0 = J1[0][2] - Bm[j][2] * J0[0], zj1 = J1[1][2] - Bm[j][2] * J0[1];
      for (int i = 0; i < 3; ++i) {
        const cx v = (wq * sb) * (cxx * (f[i][0] * in[0] + f[i][1] * in[1]) - czz * (f[i][2] * in[2]) +
                                  czr * (f[i][2] * tj) - crz * (f[i][0] * zj0 + f[i][1] * zj1));
        m[2 * (3 * i + j)] = v.r;
        m[2 * (3 * i + j) + 1] = v.i;
      }
    }
    const cx l = (wq / (gt[GEO_A] * gs[GEO_A])) * (cphi * I0);
    m[18] = l.r;
    m[19] = l.i;
  }
#pragma unroll
  for (int i = 0; i < 20; ++i) m[i] = grp_sum8(m[i]);
  if (!valid || q != 0) return;
  for (int i = 0; i < 3; ++i)
    for (int j = 0; j < 3; ++j) {
      C* dst = LA + int64_t(tri_edge[3 * t + i]) * ldA + tri_edge[3 * sidx + j];
      if (sizeof(dst->x) == 4) {
        atomicAdd(reinterpret_cast<float2*>(dst), make_float2(float(m[2 * (3 * i + j)]), float(m[2 * (3 * i + j) + 1])));
      } else {
        atomicAdd(reinterpret_cast<double*>(dst), m[2 * (3 * i + j)]);
        atomicAdd(reinterpret_cast<double*>(dst) + 1, m[2 * (3 * i + j) + 1]);
      }
    }
  C* dp = LP + int64_t(t) * ldP + sidx;
  if (sizeof(dp->x) == 4) {
    atomicAdd(reinterpret_cast<float2*>(dp), make_float2(float(m[18]), float(m[19])));
  } else {
    atomicAdd(reinterpret_cast<double*>(dp), m[18]);
    atomicAdd(reinterpret_cast<double*>(dp) + 1, m[19]);
  }
}

// Per triangle: bits 0-2 / 4-6 flag vertices on the bottom / top interface of the
// objects' layer (to 1e-9 of the mesh size); the pairs touching through an
// interface among the listed blocks (t, s, 0 = bottom / 1 = top).
void mgf_touch_setup(const HostMesh& h, const MgfStackHost& H, const std::vector<RTask>& tasks, std::vector<int32_t>& onmask,
                     std::vector<int32_t>& pairs) {
  double span = 0;
  for (int d = 0; d < 3; ++d) {
    double a = 1e300, b = -1e300;
    for (int64_t v = 0; v < h.nv; ++v) {
      a = std::min(a, h.xyz[3 * v + d]);
      b = std::max(b, h.xyz[3 * v + d]);
    }
    span = std::max(span, b - a);
  }
  const double tol = 1e-9 * span;
  onmask.assign(h.nt, 0);
  std::vector<int32_t> touching;
  for (int64_t t = 0; t < h.nt; ++t) {
    int msk = 0;
    for (int i = 0; i < 3; ++i) {
      const double z = h.xyz[3 * size_t(h.tri[3 * t + i]) + 2];
      if (H.bot && std::fabs(z - H.zb) <= tol) msk |= 1 << i;
      if (H.top && std::fabs(z - H.zu) <= tol) msk |= 1 << (4 + i);
    }
    onmask[t] = msk;
    if (msk) touching.push_back(int32_t(t));
  }
  pairs.clear();
  // `touching` is sorted: each task's test and source ranges are two slices of it
  auto slice = [&](int32_t lo, int32_t n) {
    return std::make_pair(std::lower_bound(touching.begin(), touching.end(), lo),
                          std::lower_bound(touching.begin(), touching.end(), lo + n));
  };
  for (const RTask& k : tasks) {
    const auto ta = slice(k.t0, k.ntest), tb = slice(k.s0, k.nsrc);
    for (auto ia = ta.first; ia != ta.second; ++ia) {
      const int32_t a = *ia;
      for (auto ib = tb.first; ib != tb.second; ++ib) {
        const int32_t b = *ib;
        for (int plane = 0; plane < 2; ++plane) {
          const int sh = plane ? 4 : 0;
          bool hit = false;
          for (int i = 0; i < 3 && !hit; ++i)
            for (int j = 0; j < 3 && !hit; ++j)
              hit = ((onmask[a] >> (sh + i)) & 1) && ((onmask[b] >> (sh + j)) & 1) && h.tri[3 * size_t(a) + i] == h.tri[3 * size_t(b) + j];
          if (hit) {
            pairs.push_back(a);
            pairs.push_back(b);
            pairs.push_back(plane);
          }
        }
      }
    }
  }
}

template <class C>
void mgf_fill_reflected(const sldm_mesh* m, const MgfStackHost& H, double omega, const MgfTables& T,
                        const std::vector<RTask>& tasks, void* LA, int64_t ldA, void* LP, int64_t ldP, cudaStream_t s) {
  if (tasks.empty()) return;
  const DevStack S = dev_stack(H, omega);
  ScopedTimer tm("fill_reflected", s);
  ReflArgs P{};
  {
    const std::complex<double> el = H.eps[H.l];
    const double mur = H.mu[H.l], k0 = omega / C0_;
    const std::complex<double> k = k0 * std::sqrt(mur * el);
    auto put = [](std::complex<double> z) { return cx{z.real(), z.imag()}; };
    const std::complex<double> gue(T.Q.gue.r, T.Q.gue.i), gde(T.Q.gde.r, T.Q.gde.i);
    const double guh = T.Q.guh.r, gdh = T.Q.gdh.r;  // real: permeabilities are
    P.k = put(k);
    P.ys = k.real() * (WAVE_N / (2.0 * PI));
    P.ye = k.imag() * (WAVE_N * 1.4426950408889634074);
    P.zu2 = 2 * H.zu;
    P.zb2 = 2 * H.zb;
    P.kxx_u = mur * guh;
    P.kxx_d = mur * gdh;
    P.kph_u = put(gue / el);
    P.kph_d = put(gde / el);
    P.kzz_u = put(mur * (guh - 2.0 * gue));
    P.kzz_d = put(mur * (gdh - 2.0 * gde));
    P.kzr_u = put(mur * (gue - guh));
    P.kzr_d = put(mur * (gde - gdh));
    P.nr = T.nr;
    P.ns = T.ns;
    P.nd = T.nd;
    // (log rho - lr0) (nr - 1) / (lr1 - lr0) with log rho = log2(rho^2) log(2) / 2
    const double sx = (T.nr - 1) / (T.lr1 - T.lr0);
    P.fx1 = 0.5 * std::log(2.0) * sx;
    P.fx0 = -T.lr0 * sx;
    P.s0 = T.s0;
    P.ss = T.s1 > T.s0 ? (T.ns - 1) / (T.s1 - T.s0) : 0.0;
    P.sd = T.d1 > 0 ? (T.nd - 1) / T.d1 : 0.0;
    P.rmin2 = std::exp(2 * T.lr0);
    P.inv_rmin = std::exp(-T.lr0);
  }
  DBuf<double2> ca, cb;
  auto cells = [&](const DBuf<double2>& t, int ny, DBuf<double2>& c) {
    const int n = (T.nr - 1) * ny * CELL_C;
    c.alloc(size_t(n) * 4);
    mgf_cells_kernel<<<(n + 255) / 256, 256, 0, s>>>(t.p, T.nr, ny, c.p), ::sldm::count_launch();
  };
  cells(T.A, T.ns, ca);
  if (T.hasB) cells(T.B, T.nd, cb);
  P.ca = ca.p;
  P.cb = cb.p;
  std::vector<int32_t> onmask, pairs;
  mgf_touch_setup(m->h, H, tasks, onmask, pairs);
  DBuf<RTask> dt;
  DBuf<int32_t> dm, dp;
  dt.upload(tasks, s);
  dm.upload(onmask, s);
  int64_t most = 0;
  double pairs_total = 0;
  for (const RTask& k : tasks) {
    most = std::max(most, int64_t(k.ntest) * k.nsrc);
    const bool sym = k.t0 == k.s0 && k.ntest == k.nsrc;
    pairs_total += sym ? 0.5 * k.ntest * (k.ntest + 1.0) : double(k.ntest) * k.nsrc;
  }
  {
    ScopedTimer tb("fill_reflected_bulk", s);
    timer_units("fill_reflected_bulk", 36.0 * pairs_total);
    const dim3 grid(unsigned((most + 127) / 128), unsigned(tasks.size()));
    auto go = [&](auto kernel) {
      kernel<<<grid, 128, 0, s>>>(dt.p, m->d.geo.p, m->d.tri_edge.p, m->d.tri.p, dm.p, P, (C*)LA, ldA, (C*)LP, ldP),
          ::sldm::count_launch();
    };
    if (H.top && H.bot) go(fill_reflected_kernel<C, true, true>);
    else if (H.top) go(fill_reflected_kernel<C, true, false>);
    else go(fill_reflected_kernel<C, false, true>);
    SLDM_CUDA(cudaGetLastError());
  }
  const int np = int(pairs.size() / 3);
  if (np > 0) {
    std::vector<double> x, w;
    gauss_legendre(MGF_DUFFY_N, x, w);
    for (int i = 0; i < MGF_DUFFY_N; ++i) {
      x[i] = 0.5 * (x[i] + 1);
      w[i] = 0.5 * w[i];
    }
    SLDM_CUDA(cudaMemcpyToSymbol(c_duffy_x, x.data(), sizeof(double) * MGF_DUFFY_N));
    SLDM_CUDA(cudaMemcpyToSymbol(c_duffy_w, w.data(), sizeof(double) * MGF_DUFFY_N));
    dp.upload(pairs, s);
    const int64_t threads = int64_t(np) * 8;
    fill_reflected_touch<C><<<unsigned((threads + 127) / 128), 128, 0, s>>>(dp.p, np, m->d.geo.p, m->d.xyz.p, m->d.tri.p,
                                                                            m->d.tri_edge.p, S, T.Q, (C*)LA, ldA, (C*)LP, ldP),
        ::sldm::count_launch();
    SLDM_CUDA(cudaGetLastError());
  }
  // the uploads above are released at scope exit: finish their readers first
  SLDM_CUDA(cudaStreamSynchronize(s));
}

// ---------------------------------------------------------------- stack helpers (host)
MgfStatic mgf_static(const MgfStackHost& H) {
  MgfStatic Q{};
  const int L = int(H.eps.size()), l = H.l;
  const std::complex<double> el = H.eps[l];
  const double ml = H.mu[l];
  auto pair = [&](int j, std::complex<double>* ge, double* gh) {
    *ge = (el - H.eps[j]) / (el + H.eps[j]);
    *gh = (H.mu[j] - ml) / (H.mu[j] + ml);
  };
  std::complex<double> gue = 0, gde = 0;
  double guh = 0, gdh = 0;
  if (l > 0) pair(l - 1, &gue, &guh);
  if (l < L - 1) pair(l + 1, &gde, &gdh);
  else if (H.pec) {
    gde = -1.0;
    gdh = -1.0;
  }
  Q.gue = {gue.real(), gue.imag()};
  Q.gde = {gde.real(), gde.imag()};
  Q.guh = {guh, 0.0};
  Q.gdh = {gdh, 0.0};
  return Q;
}

// Normal-incidence plane wave through the stack: E_x = a e^{+j k (z - zref)} + c e^{-j k (z - zref)} in layer l.
// Oblique plane wave through the stack, incident from the upper half-space.  The
// transverse wavevector kt = k0 (khat_x, khat_y) is common to all layers; with
// rho = kt / |kt| (at normal incidence the transverse direction of pol) and
// phi = z x rho the field splits into TE (E along phi, line impedance
// w mu0 mu_i / k_z,i) and TM (H along phi, impedance k_z,i / (w eps0 eps_i)).  For each,
// the transverse E is a transmission line in z: in layer i it is
// a e^{+j k_z (z - zref)} + c e^{-j k_z (z - zref)}, c / a at the layer's bottom the
// reflection coefficient looking down, continuous across every interface.  In the
// objects' layer E = e^{-j kt.r} [phi V_TE + rho V_TM + z (|kt| / k_z)(a_TM e^+ - c_TM e^-)].
void mgf_plane_wave(const MgfStackHost& H, const std::vector<double>& thick, double z_top, double omega, const double* khat,
                    const double* pol, double rec[PW_REC]) {
  typedef std::complex<double> C;
  const int L = int(H.eps.size());
  const double k0 = omega / C0_;
  const double ktx = k0 * khat[0], kty = k0 * khat[1];
  const double krho = std::hypot(ktx, kty);
  double rx, ry;
  if (krho > 1e-12 * k0) {
    rx = ktx / krho;
    ry = kty / krho;
  } else {
    const double n = std::hypot(pol[0], pol[1]);
    rx = n > 0 ? pol[0] / n : 1.0;
    ry = n > 0 ? pol[1] / n : 0.0;
  }
  const double px = -ry, py = rx;  // phi = z x rho
  std::vector<C> kz(L), Z(L), down(L);
  std::vector<bool> finite(L);
  for (int i = 0; i < L; ++i) {
    C q = std::sqrt(C(k0 * k0) * H.eps[i] * H.mu[i] - C(krho * krho));
    if (q.imag() > 0) q = -q;
    kz[i] = q;
    finite[i] = i > 0 && (H.pec || i < L - 1);
  }
  for (int pt = 0; pt < 2; ++pt) {  // 0: TE, 1: TM
    for (int i = 0; i < L; ++i)
      Z[i] = pt == 0 ? C(omega * MU0_ * H.mu[i]) / kz[i] : kz[i] / (omega * EPS0_ * H.eps[i]);
    down[L - 1] = H.pec ? C(-1) : C(0);
    for (int i = L - 2; i >= 0; --i) {
      const C f = (Z[i + 1] - Z[i]) / (Z[i + 1] + Z[i]);
      const C ph = finite[i + 1] ? down[i + 1] * std::exp(C(0, -2) * kz[i + 1] * thick[i + 1]) : C(0);
      down[i] = (f + ph) / (C(1) + f * ph);
    }
    const double v0 = pt == 0 ? pol[0] * px + pol[1] * py : pol[0] * rx + pol[1] * ry;
    C a = v0 * std::exp(C(0, 1) * kz[0] * z_top), c = a * down[0];
    C v = a + c;
    for (int i = 1; i <= H.l; ++i) {
      const C gtop = finite[i] ? down[i] * std::exp(C(0, -2) * kz[i] * thick[i]) : C(0);
      a = v / (C(1) + gtop);
      c = a * gtop;
      if (finite[i]) v = a * std::exp(C(0, -1) * kz[i] * thick[i]) + c * std::exp(C(0, 1) * kz[i] * thick[i]);
    }
    rec[PW_A + 4 * pt] = a.real();
    rec[PW_A + 4 * pt + 1] = a.imag();
    rec[PW_A + 4 * pt + 2] = c.real();
    rec[PW_A + 4 * pt + 3] = c.imag();
  }
  // at normal incidence pol.rho carries the whole wave, so the TM form holds with krho = 0
  rec[PW_KT] = ktx;
  rec[PW_KT + 1] = kty;
  rec[PW_RHO] = rx;
  rec[PW_RHO + 1] = ry;
  rec[PW_KZ] = kz[H.l].real();
  rec[PW_KZ + 1] = kz[H.l].imag();
  rec[PW_KRHO] = krho;
  rec[PW_ZREF] = H.l == 0 ? z_top : H.zu;
}

template void mgf_fill_reflected<float2>(const sldm_mesh*, const MgfStackHost&, double, const MgfTables&,
                                         const std::vector<RTask>&, void*, int64_t, void*, int64_t, cudaStream_t);
template void mgf_fill_reflected<double2>(const sldm_mesh*, const MgfStackHost&, double, const MgfTables&,
                                          const std::vector<RTask>&, void*, int64_t, void*, int64_t, cudaStream_t);

}  // namespace sldm
