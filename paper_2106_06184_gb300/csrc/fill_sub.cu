// Good-conductor fill (Sec. II-B: inside highly conductive objects the entries
// need integration that follows the decay of G over a skin depth).  A source
// triangle with an edge longer than 1/|Im k| is bisected through the midpoint
// of its longest edge, recursively, until no child has an edge longer than
// 1/|Im k|, and the 6-point rule runs on each child; the rules are built on the
// host per source.  Touching pairs extract 1/(4 pi R) in closed form (and
// -k^2 R/(8 pi) as well for an unsplit source, as the unsplit kernels do); for
// Kbar the static grad 1/(4 pi R) is extracted as always.  Pairs whose bounding
// spheres are farther apart than 40/|Im k| are dropped (G has decayed below e^-40).
//
// Pairs that do not touch (all but ~15 per triangle): fill_split_bulk, FP64-pipe
// bound like the unsplit bulk fill and built from the same moments (fill_dev.cuh).
// Touching pairs: one warp per pair, the lanes stride over the 6 x (points of the
// source's rule) (test point, source point) pairs, lanes 0..5 add the closed
// forms of test point q = lane, the moments are summed with shuffles, and lane 0
// scatters the 3x3 local block.  Everything is FP64; the destination precision is R.
#include <algorithm>
#include <string>
#include <vector>

#include "fill_dev.cuh"

namespace sldm {

constexpr double R8_CUTOFF = 40.0;
constexpr int SUB_MAX_CHILDREN = 4096;  // most children of one split source
constexpr double SPLIT_TIE = 1e-9;      // edges within this relative distance of the longest count as longest

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// (exp(-j k R) - 1)/(4 pi R), Taylor series for |kR| < 0.05
__device__ cd green_smooth1(cd k, double R) {
  const double ax = sqrt(k.r * k.r + k.i * k.i) * R;
  if (ax < 0.05) {
    const cd mjk = {k.i, -k.r};  // -j k
    cd p = mjk, acc = mjk;
    double Rp = 1.0, fact = 1.0;
    for (int n = 2; n <= 11; ++n) {
      p = cmul(p, mjk);
      Rp *= R;
      fact *= n;
      acc.r += p.r * Rp / fact;
      acc.i += p.i * Rp / fact;
    }
    return {acc.r * INV4PI, acc.i * INV4PI};
  }
  double sn, cn;
  sincos(k.r * R, &sn, &cn);
  const double ex = exp(k.i * R);
  return {(ex * cn - 1.0) * INV4PI / R, -ex * sn * INV4PI / R};
}

__device__ __forceinline__ void src_point(const SrcPoint& b, const double ev[3][3], double rp[3]) {
  for (int d = 0; d < 3; ++d) rp[d] = b.x * ev[0][d] + b.y * ev[1][d] + b.z * ev[2][d];
}

// ---------------------------------------------------------------- pairs that do not touch
// A CTA takes one block of SB sources against TB test triangles, one test after the
// other.  Sources are listed by the size of their rule, so the groups of 8 lanes
// of a warp, one per pair, run alike; a pair beyond the cutoff or touching is left
// out before it is given a group.  A lane takes every 8th point of the source's
// rule against all 6 test points; the 9 moments are summed over the group by a
// transposing exchange (21 additions) and left in shared memory, and then one lane
// per pair contracts and scatters them, so that those ~450 (Kbar) operations run
// with full warps.  Bound by the FP64 pipe, ~70 operations per evaluation.  Against one
// warp per pair (20 moments of r and r', 36 units on 32 lanes, bounding radii and the
// contraction per pair), the 2,048-triangle copper wire at 3 GHz: Kbar 851 -> 166 ms,
// L 239 -> 73 ms.
constexpr int SPLIT_THREADS = 128, SPLIT_SB = 64, SPLIT_TB = 8;

struct SplitTab {
  const int32_t* order;  // sources by rule size
  const int32_t* off;    // a source's points: pts[off[s] .. off[s + 1])
  const SrcPoint* pts;
};

// sum over groups of 8 lanes: lane l & 7 receives the totals of v[3 (l & 7) .. + 2]
template <int O, int N>
__device__ __forceinline__ void grp_fold(double (&v)[24], int lane) {
  const bool up = lane & O;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double send = up ? v[i] : v[i + N];
    const double keep = up ? v[i + N] : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
  }
}
__device__ __forceinline__ void grp_tsum8(double (&v)[24], int lane) {
  grp_fold<4, 12>(v, lane);
  grp_fold<2, 6>(v, lane);
  grp_fold<1, 3>(v, lane);
}

// GRAD: Kbar (sources: children), else L.  TASK: KTask or LTask.
template <class R, bool GRAD, class TASK>
__global__ void __launch_bounds__(SPLIT_THREADS, 3) fill_split_bulk(TASK tk, SplitTab rules, const double* __restrict__ geo,
                                                                    const double* __restrict__ sgeo, const double* __restrict__ rad,
                                                                    const double* __restrict__ srad, const int32_t* __restrict__ tri,
                                                                    const int32_t* __restrict__ tri_edge,
                                                                    const int32_t* __restrict__ src_edge) {
  constexpr double A1 = 0.108103018168070, B1 = 0.445948490915965, W1 = 0.223381589678011;
  constexpr double A2 = 0.816847572980459, B2 = 0.091576213509771, W2 = 0.109951743655322;
  __shared__ WaveTab tab;
  __shared__ double mom[SPLIT_SB][25];  // 18 used; odd stride
  __shared__ int32_t act[SPLIT_SB];
  __shared__ int nact;
  wave_tab_fill(tab, true);
  const int lane = threadIdx.x & 31, g8 = threadIdx.x & 7;
  const int sb = blockIdx.y * SPLIT_SB;
  int src0, nsrc;
  if constexpr (GRAD) src0 = tk.c0, nsrc = tk.nsrc;
  else src0 = tk.s0, nsrc = tk.nsrc;
  const double kr = tk.kr, ki = tk.ki;
  const double ys = kr * (WAVE_N / (2.0 * PI)), ye = ki * (WAVE_N * 1.4426950408889634074);
  for (int tt = 0; tt < SPLIT_TB; ++tt) {
    const int tl = blockIdx.x * SPLIT_TB + tt;
    if (tl >= tk.ntest) break;
    const int t = tk.t0 + tl;
    const double* gt = geo + size_t(t) * GEO_STRIDE;
    if (threadIdx.x == 0) nact = 0;
    __syncthreads();  // tables, and the last test's moments are consumed
    if (threadIdx.x < SPLIT_SB && sb + int(threadIdx.x) < nsrc) {
      const int s = src0 + rules.order[sb + threadIdx.x];
      bool use = true;
      if constexpr (GRAD) {
        const int par = s / 6, kk = s % 6, pp = kk / 2;
        const int32_t cv = tri[3 * par + ((kk & 1) ? (pp + 1) % 3 : pp)], ce = tri_edge[3 * par + (pp + 2) % 3];
        use = par != t;  // a child of the test triangle is coplanar: Kbar = 0
        for (int i = 0; i < 3; ++i) use &= tri[3 * t + i] != cv && tri_edge[3 * t + i] != ce;
      } else {
        for (int i = 0; i < 3; ++i)
          for (int j = 0; j < 3; ++j) use &= tri[3 * t + i] != tri[3 * s + j];
      }
      const double* gs = sgeo + size_t(s) * GEO_STRIDE;
      const double dx = gt[GEO_C] - gs[GEO_C], dy = gt[GEO_C + 1] - gs[GEO_C + 1], dz = gt[GEO_C + 2] - gs[GEO_C + 2];
      if (fabs(ki) * (sqrt(dx * dx + dy * dy + dz * dz) - rad[t] - srad[s]) > R8_CUTOFF) use = false;
      if (use) act[atomicAdd(&nact, 1)] = s;
    }
    __syncthreads();
    const int na = nact;
    for (int a0 = 0; a0 < na; a0 += SPLIT_THREADS / 8) {
      const int a = a0 + int(threadIdx.x) / 8;
      double v[24];
#pragma unroll
      for (int i = 0; i < 24; ++i) v[i] = 0.0;
      if (a < na) {
        const int s = act[a], sl = s - src0;
        const double* gs = sgeo + size_t(s) * GEO_STRIDE;
        const double d0 = gt[GEO_C] - gs[GEO_C], d1 = gt[GEO_C + 1] - gs[GEO_C + 1], d2 = gt[GEO_C + 2] - gs[GEO_C + 2];
        double av[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) av[i] = gs[GEO_AV + i];
        const int p1 = rules.off[sl + 1];
        for (int p = rules.off[sl] + g8; p < p1; p += 8) {
          const SrcPoint sp = rules.pts[p];
          // r - r' = dc + rho_q - r'_local, r'_local = - sum lambda_v a_v
          const double x = fma(sp.x, av[0], fma(sp.y, av[3], fma(sp.z, av[6], d0)));
          const double y = fma(sp.x, av[1], fma(sp.y, av[4], fma(sp.z, av[7], d1)));
          const double z = fma(sp.x, av[2], fma(sp.y, av[5], fma(sp.z, av[8], d2)));
          double gr[6], gi[6];
#pragma unroll
          for (int q = 0; q < 6; ++q) {
            const double dx = x + gt[GEO_RHO + 3 * q], dy = y + gt[GEO_RHO + 3 * q + 1], dz = z + gt[GEO_RHO + 3 * q + 2];
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const double ir = rsqrt_pos(r2), Rr = r2 * ir;
            double c, sn;
            wave_cis(tab, ys * Rr, c, sn);
            const double e = wave_exp2(tab, ye * Rr);
            if constexpr (GRAD) {
              const double am = -(ir * ir) * (ir * e), ai = kr * Rr, ar = fma(-ki, Rr, 1.0);
              gr[q] = am * fma(ai, sn, ar * c);
              gi[q] = am * fma(ai, c, -ar * sn);
            } else {
              const double am = ir * e;
              gr[q] = am * c;
              gi[q] = -am * sn;
            }
          }
          const double tr = W1 * B1 * (gr[0] + gr[1] + gr[2]) + W2 * B2 * (gr[3] + gr[4] + gr[5]);
          const double ti = W1 * B1 * (gi[0] + gi[1] + gi[2]) + W2 * B2 * (gi[3] + gi[4] + gi[5]);
          const double wx = sp.w * sp.x, wy = sp.w * sp.y, wz = sp.w * sp.z;
#pragma unroll
          for (int u = 0; u < 3; ++u) {
            const double lr = fma(W1 * (A1 - B1), gr[u], fma(W2 * (A2 - B2), gr[u + 3], tr));
            const double li = fma(W1 * (A1 - B1), gi[u], fma(W2 * (A2 - B2), gi[u + 3], ti));
            v[3 * u] = fma(wx, lr, v[3 * u]);
            v[3 * u + 1] = fma(wy, lr, v[3 * u + 1]);
            v[3 * u + 2] = fma(wz, lr, v[3 * u + 2]);
            v[9 + 3 * u] = fma(wx, li, v[9 + 3 * u]);
            v[10 + 3 * u] = fma(wy, li, v[10 + 3 * u]);
            v[11 + 3 * u] = fma(wz, li, v[11 + 3 * u]);
          }
        }
      }
      __syncwarp();
      grp_tsum8(v, lane);
      if (a < na)
#pragma unroll
        for (int i = 0; i < 3; ++i) mom[a][3 * g8 + i] = v[i];
    }
    __syncthreads();
    // one lane per pair
    if (int(threadIdx.x) < na) {
      const int s = act[threadIdx.x];
      const double* gs = sgeo + size_t(s) * GEO_STRIDE;
      double Nr[9], Ni[9], av[9], bv[9], dc[3];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        Nr[i] = mom[threadIdx.x][i];
        Ni[i] = mom[threadIdx.x][9 + i];
        av[i] = gt[GEO_AV + i];
        bv[i] = gs[GEO_AV + i];
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) dc[d] = gt[GEO_C + d] - gs[GEO_C + d];
      if constexpr (GRAD) {
        contract_K(Nr, Ni, av, bv, dc, [&](int i, int j, double vr, double vi) {
          const double sc = half_sign<double>(gt[GEO_SIG + i]) * (half_sign<double>(gs[GEO_SIG + j]) * INV4PI);
          add_d<R>(tk.Kb, int64_t(tri_edge[3 * t + i] - tk.e_row0) * tk.ld + (src_edge[3 * s + j] - tk.b_col0), vr * sc, vi * sc);
        });
      } else {
        const double Sr = sum9(Nr), Si = sum9(Ni);
        if (tk.A)
          contract_L(Nr, Ni, Sr, Si, av, bv, [&](int i, int j, double vr, double vi) {
            const double sc = half_sign<double>(gt[GEO_SIG + i]) * (half_sign<double>(gs[GEO_SIG + j]) * INV4PI);
            const cd out = cmul({vr * sc, vi * sc}, {tk.sAr, tk.sAi});
            add_d<R>(tk.A, int64_t(tri_edge[3 * t + i] - tk.e_row0) * tk.ldA + (src_edge[3 * s + j] - tk.e_col0), out.r, out.i);
          });
        if (tk.P) {  // 1/(A A') against the areas of the two integrals
          const cd out = cmul({Sr * INV4PI, Si * INV4PI}, {tk.sPr, tk.sPi});
          M<R>::store(tk.P, int64_t(t - tk.t_row0) * tk.ldP + (s - tk.t_col0), out.r, out.i);
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- L^A, L^phi, touching pairs
template <class R>
__global__ void __launch_bounds__(256) fill_L_split(LTask tk, const int32_t* __restrict__ pa, const int32_t* __restrict__ pb,
                                                    int npairs, const int32_t* __restrict__ soff,
                                                    const SrcPoint* __restrict__ spts,
                                                    const double* __restrict__ geo, const double* __restrict__ xyz,
                                                    const int32_t* __restrict__ tri, const int32_t* __restrict__ tri_edge) {
  const int64_t pair = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (pair >= npairs) return;  // whole warps
  const int t = pa[pair], s = pb[pair];
  if (t < tk.t0 || t >= tk.t0 + tk.ntest || s < tk.s0 || s >= tk.s0 + tk.nsrc) return;
  const double* gt = geo + size_t(t) * GEO_STRIDE;
  const double* gs = geo + size_t(s) * GEO_STRIDE;
  const int32_t sv[3] = {tri[3 * s], tri[3 * s + 1], tri[3 * s + 2]};
  const double* ps[3] = {xyz + 3 * sv[0], xyz + 3 * sv[1], xyz + 3 * sv[2]};
  const SrcPoint* rule = spts + soff[s - tk.s0];
  const int nu = soff[s - tk.s0 + 1] - soff[s - tk.s0];
  const bool split = nu > 6;
  const double As = gs[GEO_A];
  double ev[3][3], dc[3];
  for (int i = 0; i < 3; ++i)
    for (int d = 0; d < 3; ++d) ev[i][d] = ps[i][d] - gs[GEO_C + d];
  for (int d = 0; d < 3; ++d) dc[d] = gt[GEO_C + d] - gs[GEO_C + d];
  const cd k = {tk.kr, tk.ki};
  // m: M0 (0,1), Mq (2..7), Ms (8..13), Mqs (14,15)
  double m[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) m[i] = 0.0;
  // unit u = (source point u / 6, test point u % 6): 36 units even when unsplit
  for (int u = lane; u < 6 * nu; u += 32) {
    const int pnt = u / 6, q = u - 6 * pnt;
    const SrcPoint sp = rule[pnt];
    double rp[3];
    src_point(sp, ev, rp);
    const double ws = As * sp.w;
    const double* rq = gt + GEO_RHO + 3 * q;
    const double D0 = dc[0] + rq[0] - rp[0], D1 = dc[1] + rq[1] - rp[1], D2 = dc[2] + rq[2] - rp[2];
    const double r2 = D0 * D0 + D1 * D1 + D2 * D2;
    cd g = split ? green_smooth1(k, sqrt(r2)) : green_smooth(k, sqrt(r2));
    const double w = gt[GEO_W + q] * ws;
    g.r *= w;
    g.i *= w;
    const double qs = rq[0] * rp[0] + rq[1] * rp[1] + rq[2] * rp[2];
    m[0] += g.r;
    m[1] += g.i;
    for (int d = 0; d < 3; ++d) {
      m[2 + 2 * d] += g.r * rq[d];
      m[3 + 2 * d] += g.i * rq[d];
      m[8 + 2 * d] += g.r * rp[d];
      m[9 + 2 * d] += g.i * rp[d];
    }
    m[14] += g.r * qs;
    m[15] += g.i * qs;
  }
  if (lane < 6) {
    const int q = lane;
    const double* rq = gt + GEO_RHO + 3 * q;
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = gt[GEO_C + d] + rq[d];
    Pot P;
    potentials(r, ps[0], ps[1], ps[2], P);
    const cd k2 = cmul(k, k);
    const double two = split ? 0.0 : 1.0;  // the k^2 R term is extracted only when unsplit
    cd A = {INV4PI * P.inv_r - two * k2.r * 0.5 * INV4PI * P.r, -two * k2.i * 0.5 * INV4PI * P.r};
    cd Bv[3];
    for (int d = 0; d < 3; ++d) {
      const double off = P.rho[d] - gs[GEO_C + d];
      const double s1 = P.por[d] + off * P.inv_r;
      const double sR = P.pr[d] + off * P.r;
      Bv[d] = {INV4PI * s1 - two * k2.r * 0.5 * INV4PI * sR, -two * k2.i * 0.5 * INV4PI * sR};
    }
    const double w = gt[GEO_W + q];
    m[0] += w * A.r;
    m[1] += w * A.i;
    for (int d = 0; d < 3; ++d) {
      m[2 + 2 * d] += w * A.r * rq[d];
      m[3 + 2 * d] += w * A.i * rq[d];
      m[8 + 2 * d] += w * Bv[d].r;
      m[9 + 2 * d] += w * Bv[d].i;
      m[14] += w * rq[d] * Bv[d].r;
      m[15] += w * rq[d] * Bv[d].i;
    }
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) m[i] = warp_sum(m[i]);
  if (lane != 0) return;
  const cd m0 = {m[0], m[1]}, mqs = {m[14], m[15]};
  cd mq[3], ms[3];
  for (int d = 0; d < 3; ++d) {
    mq[d] = {m[2 + 2 * d], m[3 + 2 * d]};
    ms[d] = {m[8 + 2 * d], m[9 + 2 * d]};
  }
  if (tk.A) {
    for (int i = 0; i < 3; ++i) {
      const double* a = gt + GEO_AV + 3 * i;
      for (int j = 0; j < 3; ++j) {
        const double* b = gs + GEO_AV + 3 * j;
        const double ab = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
        cd v = mqs;
        for (int d = 0; d < 3; ++d) {
          v.r += a[d] * ms[d].r + b[d] * mq[d].r;
          v.i += a[d] * ms[d].i + b[d] * mq[d].i;
        }
        v.r += ab * m0.r;
        v.i += ab * m0.i;
        const double sc = gt[GEO_SIG + i] * gs[GEO_SIG + j];
        const cd out = cmul({v.r * sc, v.i * sc}, {tk.sAr, tk.sAi});
        add_d<R>(tk.A, int64_t(tri_edge[3 * t + i] - tk.e_row0) * tk.ldA + (tri_edge[3 * s + j] - tk.e_col0), out.r, out.i);
      }
    }
  }
  if (tk.P) {
    const double sc = 1.0 / (gt[GEO_A] * gs[GEO_A]);
    const cd out = cmul({m0.r * sc, m0.i * sc}, {tk.sPr, tk.sPi});
    M<R>::store(tk.P, int64_t(t - tk.t_row0) * tk.ldP + (s - tk.t_col0), out.r, out.i);
  }
}

// ---------------------------------------------------------------- Kbar (primal test x barycentric child), touching pairs
template <class R>
__global__ void __launch_bounds__(256) fill_K_split(KTask tk, const int32_t* __restrict__ pa, const int32_t* __restrict__ pc,
                                                    int npairs, const int32_t* __restrict__ soff,
                                                    const SrcPoint* __restrict__ spts,
                                                    const double* __restrict__ geo,
                                                    const double* __restrict__ bgeo, const double* __restrict__ xyz,
                                                    const int32_t* __restrict__ tri, const int32_t* __restrict__ tri_edge,
                                                    const int32_t* __restrict__ btri_edge) {
  const int64_t pair = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (pair >= npairs) return;
  const int t = pa[pair], cg = pc[pair];
  if (t < tk.t0 || t >= tk.t0 + tk.ntest || cg < tk.c0 || cg >= tk.c0 + tk.nsrc) return;
  const int par = cg / 6, kk = cg % 6;
  const double* gt = geo + size_t(t) * GEO_STRIDE;
  const double* gs = bgeo + size_t(cg) * GEO_STRIDE;
  // child vertices rebuilt from the parent: (a, m_ab, g) (m_ab, b, g) (b, m_bc, g) (m_bc, c, g) (c, m_ca, g) (m_ca, a, g)
  const double* a = xyz + 3 * tri[3 * par];
  const double* b = xyz + 3 * tri[3 * par + 1];
  const double* c = xyz + 3 * tri[3 * par + 2];
  double V[7][3];
  for (int d = 0; d < 3; ++d) {
    V[0][d] = a[d]; V[1][d] = b[d]; V[2][d] = c[d];
    V[3][d] = 0.5 * (a[d] + b[d]); V[4][d] = 0.5 * (b[d] + c[d]); V[5][d] = 0.5 * (c[d] + a[d]);
    V[6][d] = (a[d] + b[d] + c[d]) / 3.0;
  }
  const int cvt[6][3] = {{0, 3, 6}, {3, 1, 6}, {1, 4, 6}, {4, 2, 6}, {2, 5, 6}, {5, 0, 6}};
  const double* ps[3] = {V[cvt[kk][0]], V[cvt[kk][1]], V[cvt[kk][2]]};
  const SrcPoint* rule = spts + soff[cg - tk.c0];
  const int nu = soff[cg - tk.c0 + 1] - soff[cg - tk.c0];
  const double As = gs[GEO_A];
  double ev[3][3], dc[3];
  for (int i = 0; i < 3; ++i)
    for (int d = 0; d < 3; ++d) ev[i][d] = ps[i][d] - gs[GEO_C + d];
  for (int d = 0; d < 3; ++d) dc[d] = gt[GEO_C + d] - gs[GEO_C + d];
  const cd k = {tk.kr, tk.ki};
  // m: P1 (0,1), P2 (2..7), X (8..13), S (14..19)
  double m[20];
#pragma unroll
  for (int i = 0; i < 20; ++i) m[i] = 0.0;
  // unit u = (source point u / 6, test point u % 6)
  for (int u = lane; u < 6 * nu; u += 32) {
    const int pnt = u / 6, q = u - 6 * pnt;
    const SrcPoint sp = rule[pnt];
    double rp[3];
    src_point(sp, ev, rp);
    const double ws = As * sp.w;
    const double* rq = gt + GEO_RHO + 3 * q;
    const double D[3] = {dc[0] + rq[0] - rp[0], dc[1] + rq[1] - rp[1], dc[2] + rq[2] - rp[2]};
    const double r2 = D[0] * D[0] + D[1] * D[1] + D[2] * D[2];
    cd g1 = grad_smooth(k, sqrt(r2));
    const double w = gt[GEO_W + q] * ws;
    g1.r *= w;
    g1.i *= w;
    const double cr[3] = {D[1] * rp[2] - D[2] * rp[1], D[2] * rp[0] - D[0] * rp[2], D[0] * rp[1] - D[1] * rp[0]};
    const double xq[3] = {rq[1] * D[2] - rq[2] * D[1], rq[2] * D[0] - rq[0] * D[2], rq[0] * D[1] - rq[1] * D[0]};
    const double p1 = rq[0] * cr[0] + rq[1] * cr[1] + rq[2] * cr[2];
    m[0] += g1.r * p1;
    m[1] += g1.i * p1;
    for (int d = 0; d < 3; ++d) {
      m[2 + 2 * d] += g1.r * cr[d];
      m[3 + 2 * d] += g1.i * cr[d];
      m[8 + 2 * d] += g1.r * xq[d];
      m[9 + 2 * d] += g1.i * xq[d];
      m[14 + 2 * d] += g1.r * D[d];
      m[15 + 2 * d] += g1.i * D[d];
    }
  }
  if (lane < 6) {
    // static part: V_s = int grad 1/(4 pi R) dS', U_s = V_s x (r - c')
    const int q = lane;
    const double* rq = gt + GEO_RHO + 3 * q;
    double r[3];
    for (int d = 0; d < 3; ++d) r[d] = gt[GEO_C + d] + rq[d];
    Pot P;
    potentials(r, ps[0], ps[1], ps[2], P);
    double vs[3], rc[3];
    for (int d = 0; d < 3; ++d) {
      vs[d] = INV4PI * P.grad[d];
      rc[d] = r[d] - gs[GEO_C + d];
    }
    const double us[3] = {vs[1] * rc[2] - vs[2] * rc[1], vs[2] * rc[0] - vs[0] * rc[2], vs[0] * rc[1] - vs[1] * rc[0]};
    const double w = gt[GEO_W + q];
    m[0] += w * (rq[0] * us[0] + rq[1] * us[1] + rq[2] * us[2]);
    const double xq[3] = {rq[1] * vs[2] - rq[2] * vs[1], rq[2] * vs[0] - rq[0] * vs[2], rq[0] * vs[1] - rq[1] * vs[0]};
    for (int d = 0; d < 3; ++d) {
      m[2 + 2 * d] += w * us[d];
      m[8 + 2 * d] += w * xq[d];
      m[14 + 2 * d] += w * vs[d];
    }
  }
#pragma unroll
  for (int i = 0; i < 20; ++i) m[i] = warp_sum(m[i]);
  if (lane != 0) return;
  const cd P1 = {m[0], m[1]};
  cd P2[3], X[3], S[3];
  for (int d = 0; d < 3; ++d) {
    P2[d] = {m[2 + 2 * d], m[3 + 2 * d]};
    X[d] = {m[8 + 2 * d], m[9 + 2 * d]};
    S[d] = {m[14 + 2 * d], m[15 + 2 * d]};
  }
  for (int i = 0; i < 3; ++i) {
    const double* av = gt + GEO_AV + 3 * i;
    cd base = P1;
    for (int d = 0; d < 3; ++d) {
      base.r += av[d] * P2[d].r;
      base.i += av[d] * P2[d].i;
    }
    const cd axs[3] = {{av[1] * S[2].r - av[2] * S[1].r, av[1] * S[2].i - av[2] * S[1].i},
                       {av[2] * S[0].r - av[0] * S[2].r, av[2] * S[0].i - av[0] * S[2].i},
                       {av[0] * S[1].r - av[1] * S[0].r, av[0] * S[1].i - av[1] * S[0].i}};
    for (int j = 0; j < 3; ++j) {
      const double* bv = gs + GEO_AV + 3 * j;
      cd v = base;
      for (int d = 0; d < 3; ++d) {
        v.r += bv[d] * (X[d].r + axs[d].r);
        v.i += bv[d] * (X[d].i + axs[d].i);
      }
      const double sc = gt[GEO_SIG + i] * gs[GEO_SIG + j];
      add_d<R>(tk.Kb, int64_t(tri_edge[3 * t + i] - tk.e_row0) * tk.ld + (btri_edge[3 * cg + j] - tk.b_col0), v.r * sc,
               v.i * sc);
    }
  }
}

// ---------------------------------------------------------------- host side
static const double kBary[6][3] = {
    {0.108103018168070, 0.445948490915965, 0.445948490915965}, {0.445948490915965, 0.108103018168070, 0.445948490915965},
    {0.445948490915965, 0.445948490915965, 0.108103018168070}, {0.816847572980459, 0.091576213509771, 0.091576213509771},
    {0.091576213509771, 0.816847572980459, 0.091576213509771}, {0.091576213509771, 0.091576213509771, 0.816847572980459}};
static const double kW[6] = {0.223381589678011, 0.223381589678011, 0.223381589678011,
                              0.109951743655322, 0.109951743655322, 0.109951743655322};

static double edge_len(const double* a, const double* b) {
  return std::sqrt((a[0] - b[0]) * (a[0] - b[0]) + (a[1] - b[1]) * (a[1] - b[1]) + (a[2] - b[2]) * (a[2] - b[2]));
}

// The source's quadrature appended to `pts`: longest-edge bisection of the
// triangle (p0, p1, p2) until no child has an edge longer than h (edge i joins
// vertices i and i + 1; the first edge within SPLIT_TIE of the longest is cut;
// the child holding the cut edge's first vertex is refined first), then the
// 6-point rule on each child.
struct Child {
  double B[3][3];  // barycentric coordinates of the child's vertices
  double f;        // area fraction
};
static void append_rule(const double* p0, const double* p1, const double* p2, double h, std::vector<SrcPoint>& pts) {
  const double* P[3] = {p0, p1, p2};
  std::vector<Child> todo(1), done;
  todo[0] = Child{{{1, 0, 0}, {0, 1, 0}, {0, 0, 1}}, 1.0};
  while (!todo.empty()) {
    const Child c = todo.back();
    todo.pop_back();
    double X[3][3];
    for (int v = 0; v < 3; ++v)
      for (int d = 0; d < 3; ++d) X[v][d] = c.B[v][0] * P[0][d] + c.B[v][1] * P[1][d] + c.B[v][2] * P[2][d];
    const double L[3] = {edge_len(X[0], X[1]), edge_len(X[1], X[2]), edge_len(X[2], X[0])};
    const double Lmax = std::max(L[0], std::max(L[1], L[2]));
    if (!(Lmax > h)) {
      done.push_back(c);
      continue;
    }
    int i = 0;
    while (!(L[i] >= (1.0 - SPLIT_TIE) * Lmax)) ++i;
    const double* a = c.B[i];
    const double* b = c.B[(i + 1) % 3];
    const double* cc = c.B[(i + 2) % 3];
    Child c1, c2;
    for (int d = 0; d < 3; ++d) {
      const double m = 0.5 * (a[d] + b[d]);
      c1.B[0][d] = m; c1.B[1][d] = b[d]; c1.B[2][d] = cc[d];
      c2.B[0][d] = a[d]; c2.B[1][d] = m; c2.B[2][d] = cc[d];
    }
    c1.f = c2.f = 0.5 * c.f;
    todo.push_back(c1);
    todo.push_back(c2);
    SLDM_REQUIRE(done.size() + todo.size() <= size_t(SUB_MAX_CHILDREN), SLDM_ENOTSUP,
                 "source triangle too large for the skin depth: more than " + std::to_string(SUB_MAX_CHILDREN) +
                     " children");
  }
  for (const Child& c : done)
    for (int j = 0; j < 6; ++j) {
      double b[3] = {0, 0, 0};
      for (int v = 0; v < 3; ++v)
        for (int d = 0; d < 3; ++d) b[d] += kBary[j][v] * c.B[v][d];
      pts.push_back(SrcPoint{b[0], b[1], b[2], c.f * kW[j]});
    }
}

static double longest_edge(const double* p0, const double* p1, const double* p2) {
  return std::max(edge_len(p0, p2), std::max(edge_len(p1, p0), edge_len(p2, p1)));
}

template <class VertexFn>
static SplitRules make_rules(int nsrc, double ki, VertexFn vertices) {
  SplitRules R;
  const double aki = std::fabs(ki);
  for (int i = 0; i < nsrc && !R.split; ++i) {
    const double* p[3];
    double store[3][3];
    vertices(i, p, store);
    R.split = aki * longest_edge(p[0], p[1], p[2]) > 1.0;
  }
  if (!R.split) return R;
  const double h = 1.0 / aki;
  R.off.reserve(size_t(nsrc) + 1);
  for (int i = 0; i < nsrc; ++i) {
    R.off.push_back(int32_t(R.pts.size()));
    const double* p[3];
    double store[3][3];
    vertices(i, p, store);
    append_rule(p[0], p[1], p[2], h, R.pts);
  }
  R.off.push_back(int32_t(R.pts.size()));
  return R;
}

SplitRules split_rules_L(const HostMesh& h, const LTask& tk) {
  return make_rules(tk.nsrc, tk.ki, [&](int i, const double* p[3], double (*)[3]) {
    const int s = tk.s0 + i;
    for (int v = 0; v < 3; ++v) p[v] = &h.xyz[3 * size_t(h.tri[3 * s + v])];
  });
}

SplitRules split_rules_K(const HostMesh& h, const KTask& tk) {
  static const int cvt[6][3] = {{0, 3, 6}, {3, 1, 6}, {1, 4, 6}, {4, 2, 6}, {2, 5, 6}, {5, 0, 6}};
  return make_rules(tk.nsrc, tk.ki, [&](int i, const double* p[3], double (*store)[3]) {
    const int cg = tk.c0 + i, par = cg / 6, kk = cg % 6;
    const double* a = &h.xyz[3 * size_t(h.tri[3 * par])];
    const double* b = &h.xyz[3 * size_t(h.tri[3 * par + 1])];
    const double* c = &h.xyz[3 * size_t(h.tri[3 * par + 2])];
    double V[7][3];
    for (int d = 0; d < 3; ++d) {
      V[0][d] = a[d]; V[1][d] = b[d]; V[2][d] = c[d];
      V[3][d] = 0.5 * (a[d] + b[d]); V[4][d] = 0.5 * (b[d] + c[d]); V[5][d] = 0.5 * (c[d] + a[d]);
      V[6][d] = (a[d] + b[d] + c[d]) / 3.0;
    }
    for (int v = 0; v < 3; ++v) {
      for (int d = 0; d < 3; ++d) store[v][d] = V[cvt[kk][v]][d];
      p[v] = store[v];
    }
  });
}

// sources of a task by rule size, largest first (mesh order among equals)
static std::vector<int32_t> by_rule_size(const SplitRules& rules) {
  std::vector<int32_t> o(rules.off.size() - 1);
  for (size_t i = 0; i < o.size(); ++i) o[i] = int32_t(i);
  std::stable_sort(o.begin(), o.end(), [&](int32_t a, int32_t b) {
    return rules.off[a + 1] - rules.off[a] > rules.off[b + 1] - rules.off[b];
  });
  return o;
}

template <class R>
void fill_L_split_task(const sldm_mesh* m, const LTask& tk, const SplitRules& rules, cudaStream_t s) {
  DBuf<int32_t> doff, dord;
  DBuf<SrcPoint> dpts;
  doff.upload(rules.off, s);
  dpts.upload(rules.pts, s);
  dord.upload(by_rule_size(rules), s);
  const DevMesh& d = m->d;
  const int np = int(m->h.touchL_a.size());
  {
    ScopedTimer tm("fill_L_split", s);
    fill_split_bulk<R, false><<<dim3((tk.ntest + SPLIT_TB - 1) / SPLIT_TB, (tk.nsrc + SPLIT_SB - 1) / SPLIT_SB), SPLIT_THREADS, 0,
                                s>>>(tk, SplitTab{dord.p, doff.p, dpts.p}, d.geo.p, d.geo.p, d.rad.p, d.rad.p, d.tri.p,
                                     d.tri_edge.p, d.tri_edge.p), ::sldm::count_launch();
    fill_L_split<R><<<unsigned((int64_t(np) * 32 + 255) / 256), 256, 0, s>>>(tk, d.touchL_a.p, d.touchL_b.p, np, doff.p, dpts.p,
                                                                            d.geo.p, d.xyz.p, d.tri.p, d.tri_edge.p),
        ::sldm::count_launch();
  }
  SLDM_CUDA(cudaGetLastError());
  SLDM_CUDA(cudaStreamSynchronize(s));
}

template <class R>
void fill_K_split_task(const sldm_mesh* m, const KTask& tk, const SplitRules& rules, cudaStream_t s) {
  DBuf<int32_t> doff, dord;
  DBuf<SrcPoint> dpts;
  doff.upload(rules.off, s);
  dpts.upload(rules.pts, s);
  dord.upload(by_rule_size(rules), s);
  const DevMesh& d = m->d;
  const int np = int(m->h.touchK_a.size());
  {
    ScopedTimer tm("fill_K_split", s);
    fill_split_bulk<R, true><<<dim3((tk.ntest + SPLIT_TB - 1) / SPLIT_TB, (tk.nsrc + SPLIT_SB - 1) / SPLIT_SB), SPLIT_THREADS, 0,
                               s>>>(tk, SplitTab{dord.p, doff.p, dpts.p}, d.geo.p, d.bgeo.p, d.rad.p, d.brad.p, d.tri.p,
                                    d.tri_edge.p, d.btri_edge.p), ::sldm::count_launch();
    fill_K_split<R><<<unsigned((int64_t(np) * 32 + 255) / 256), 256, 0, s>>>(tk, d.touchK_a.p, d.touchK_c.p, np, doff.p, dpts.p,
                                                                            d.geo.p, d.bgeo.p, d.xyz.p, d.tri.p, d.tri_edge.p,
                                                                            d.btri_edge.p), ::sldm::count_launch();
  }
  SLDM_CUDA(cudaGetLastError());
  SLDM_CUDA(cudaStreamSynchronize(s));
}

template void fill_L_split_task<float>(const sldm_mesh*, const LTask&, const SplitRules&, cudaStream_t);
template void fill_L_split_task<double>(const sldm_mesh*, const LTask&, const SplitRules&, cudaStream_t);
template void fill_K_split_task<float>(const sldm_mesh*, const KTask&, const SplitRules&, cudaStream_t);
template void fill_K_split_task<double>(const sldm_mesh*, const KTask&, const SplitRules&, cudaStream_t);

}  // namespace sldm
