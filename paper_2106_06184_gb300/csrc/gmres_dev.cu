// GMRES on the device: residuals and their norms for all columns at once, the
// Gram-Schmidt step of a small system in one launch, Givens rotations and
// convergence tests, the cycle's back substitution and update (Sec. IV).
#include <algorithm>

#include "cluster.h"
#include "dense.h"
#include "widen.cuh"

namespace sldm {

namespace {

__device__ __forceinline__ double2 zmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

template <class C>
struct Real;
template <>
struct Real<float2> {
  typedef float R;
};
template <>
struct Real<double2> {
  typedef double R;
};
template <class C>
__device__ __forceinline__ C cmake(double x, double y) {
  C c;
  c.x = decltype(c.x)(x);
  c.y = decltype(c.y)(y);
  return c;
}

__device__ __forceinline__ double warp_total(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// sum over the CTA into *out (atomic); red: one double per warp
__device__ __forceinline__ void add_norm(double v, double* red, double* out) {
  v = warp_total(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (unsigned w = 1; w < blockDim.x / 32; ++w) v += red[w];
    atomicAdd(out, v);
  }
}

// b = D b with D = diag(1, 1, l), r = b, nrm[c] += |b|^2
__global__ void __launch_bounds__(256) rhs_scale_kernel(int64_t n, int64_t n2, double l, double2* b, double2* r, double* nrm) {
  __shared__ double red[8];
  const int64_t t = int64_t(blockIdx.x) * 256 + threadIdx.x, c = blockIdx.y;
  double s = 0;
  if (t < n) {
    double2 v = b[c * n + t];
    if (t >= n2) v = make_double2(l * v.x, l * v.y);
    b[c * n + t] = v;
    r[c * n + t] = v;
    s = v.x * v.x + v.y * v.y;
  }
  add_norm(s, red, nrm + c);
}
// r = b - y, nrm[c] += |r|^2
__global__ void __launch_bounds__(256) residual_kernel(int64_t n, const double2* __restrict__ b, const double2* __restrict__ y,
                                                       double2* __restrict__ r, double* nrm) {
  __shared__ double red[8];
  const int64_t t = int64_t(blockIdx.x) * 256 + threadIdx.x, c = blockIdx.y;
  double s = 0;
  if (t < n) {
    const double2 u = b[c * n + t], v = y[c * n + t];
    const double2 d = make_double2(u.x - v.x, u.y - v.y);
    r[c * n + t] = d;
    s = d.x * d.x + d.y * d.y;
  }
  add_norm(s, red, nrm + c);
}

// a cycle starts: v_0 = r / beta, the residual vector g = (beta, 0, ..), the state
template <class CB>
__global__ void __launch_bounds__(256) cycle_start_kernel(int64_t n, CycleStart a) {
  const int c = blockIdx.y;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.st[c] = GmresState{a.it[c], 0, a.live[c], 0, a.bnorm[c], a.beta[c]};
    a.g[int64_t(c) * (a.m + 1)] = make_double2(a.beta[c], 0.0);
  }
  if (!a.live[c]) return;
  const int64_t t = int64_t(blockIdx.x) * 256 + threadIdx.x;
  if (t >= n) return;
  const double s = 1.0 / a.beta[c];
  const double2 v = a.r[c * n + t];
  reinterpret_cast<CB*>(a.v0[c])[t] = cmake<CB>(s * v.x, s * v.y);
}

// ---------------------------------------------------------------- rotations
// One warp: column k of H_r from its k + 1 projection coefficients col (shared memory)
// and h1 = h_{k+1,k}.  Rotation i maps (x_i, h_{i+1}) to (c x_i + s h_{i+1}, -conj(s) x_i +
// c h_{i+1}) = (H_i, x_{i+1}): a linear recurrence in x, so each lane composes the
// maps of its k / 32 rotations, a scan over the lanes gives every lane its first x,
// and the entries follow.  One lane walking the chain took 20 us at k ~ 20 and 60 us
// at k ~ 150.  rot (shared memory): the k earlier rotations, (c, Re s, Im s), staged by
// stage_rotations.
struct Rot {
  double c, sr, si;
};
__device__ __forceinline__ void stage_rotations(const GivensArgs& a, int r, Rot* rot) {
  const double2* cs = a.cs + int64_t(r) * a.m;
  const double2* sn = a.sn + int64_t(r) * a.m;
  for (int i = threadIdx.x; i < a.k; i += blockDim.x) rot[i] = Rot{cs[i].x, sn[i].x, sn[i].y};
}
__device__ void givens_column(const GivensArgs& a, int j, double h1, const double2* col, const Rot* rot) {
  const int r = a.on[j], lane = threadIdx.x & 31, k = a.k, m = a.m;
  double2* H = a.H + int64_t(r) * (m + 1) * m;
  double2* cs = a.cs + int64_t(r) * m;
  double2* sn = a.sn + int64_t(r) * m;
  double2* g = a.g + int64_t(r) * (m + 1);
  GmresState* st = a.st + r;
  const int seg = (k + 31) / 32, i0 = min(k, lane * seg), i1 = min(k, i0 + seg);
  double2 A = make_double2(1.0, 0.0), B = make_double2(0.0, 0.0);
  for (int i = i0; i < i1; ++i) {
    const double c = rot[i].c;
    const double2 t = make_double2(-rot[i].sr, rot[i].si);  // -conj(s)
    A = zmul(t, A);
    B = zadd(zmul(t, B), make_double2(c * col[i + 1].x, c * col[i + 1].y));
  }
  for (int o = 1; o < 32; o <<= 1) {  // inclusive scan of the maps x -> A x + B
    const double2 pa = make_double2(__shfl_up_sync(0xffffffffu, A.x, o), __shfl_up_sync(0xffffffffu, A.y, o));
    const double2 pb = make_double2(__shfl_up_sync(0xffffffffu, B.x, o), __shfl_up_sync(0xffffffffu, B.y, o));
    if (lane >= o) {
      B = zadd(zmul(A, pb), B);
      A = zmul(A, pa);
    }
  }
  const double2 xe = zadd(zmul(A, col[0]), B);  // x after this lane's rotations
  double2 x = make_double2(__shfl_up_sync(0xffffffffu, xe.x, 1), __shfl_up_sync(0xffffffffu, xe.y, 1));
  if (lane == 0) x = col[0];
  for (int i = i0; i < i1; ++i) {
    const double2 s = make_double2(rot[i].sr, rot[i].si), y = col[i + 1];
    const double c = rot[i].c;
    H[int64_t(i) * m + k] = zadd(make_double2(c * x.x, c * x.y), zmul(s, y));
    x = zadd(zmul(make_double2(-s.x, s.y), x), make_double2(c * y.x, c * y.y));
  }
  const double2 xk = make_double2(__shfl_sync(0xffffffffu, xe.x, 31), __shfl_sync(0xffffffffu, xe.y, 31));
  if (lane != 0) return;
  // the new rotation annihilates h_{k+1,k}
  const double2 gk = g[k];
  const double bnorm = st->bnorm, beta = st->beta;
  const int its = st->it + 1;
  const double ax2 = xk.x * xk.x + xk.y * xk.y, t2 = fma(h1, h1, ax2);
  const double it_ = rsqrt(t2), ia = rsqrt(ax2), t = t2 * it_;
  double2 c, sv, d;
  if (!(ax2 > 0)) {
    c = make_double2(0.0, 0.0);
    sv = make_double2(1.0, 0.0);
    d = make_double2(h1, 0.0);
  } else {
    const double2 ph = make_double2(xk.x * ia, xk.y * ia);  // x / |x|
    c = make_double2(ax2 * ia * it_, 0.0);
    sv = make_double2(ph.x * h1 * it_, ph.y * h1 * it_);
    d = make_double2(ph.x * t, ph.y * t);
  }
  const double2 gn = zmul(make_double2(-sv.x, sv.y), gk);
  const double res = sqrt(gn.x * gn.x + gn.y * gn.y);
  int live = 1;
  if (res <= a.tol * bnorm || its >= a.maxit || h1 == 0) live = 0;
  if (a.refine && res <= a.cycle * beta) live = 0;
  a.flags[r] = live;
  if (!live) st->live = 0;
  st->it = its;
  st->kused = k + 1;
  H[int64_t(k) * m + k] = d;
  H[int64_t(k + 1) * m + k] = make_double2(0.0, 0.0);
  cs[k] = c;
  sn[k] = sv;
  g[k + 1] = gn;
  g[k] = zmul(c, gk);
}

// ---------------------------------------------------------------- end of a step, separate launches
// v_{k+1} = w / h_{k+1,k} (zero once the right-hand side has stopped); the first CTA
// of a column makes the rotations instead.  A CTA that sees the state after that
// one has stopped the column writes zeros into a vector nothing reads.
template <class CB>
__global__ void __launch_bounds__(256) gmres_close_kernel(GivensArgs a, VecBatch<CB, CB> v, int64_t n) {
  extern __shared__ __align__(16) unsigned char gc_raw[];
  __shared__ double scale;
  const int j = blockIdx.y, r = a.on[j];
  const bool live = a.st[r].live != 0;
  if (blockIdx.x == 0) {
    if (!live) {
      if (threadIdx.x == 0) a.flags[r] = 0;
      return;
    }
    double2* col = reinterpret_cast<double2*>(gc_raw);
    Rot* rot = reinterpret_cast<Rot*>(col + a.k + 1);
    const double2* hr = a.dh + int64_t(r) * a.ldh;
    for (int i = threadIdx.x; i <= a.k; i += 256) col[i] = zadd(hr[i], hr[(a.m + 2) + i]);
    stage_rotations(a, r, rot);
    __syncthreads();  // staged, and every warp has read the state
    if (threadIdx.x < 32) givens_column(a, j, sqrt(a.nrm[j]), col, rot);
    return;
  }
  // once per CTA: a square root and a quotient are ~45 FP64 instructions per warp
  if (threadIdx.x == 0) scale = live && a.nrm[j] > 0 ? 1.0 / sqrt(a.nrm[j]) : 0.0;
  __syncthreads();
  const double sc = scale;
  for (int64_t t = int64_t(blockIdx.x - 1) * 256 + threadIdx.x; t < n; t += int64_t(gridDim.x - 1) * 256) {
    CB w = v.y[j][t];
    w.x = decltype(w.x)(widen(w.x) * sc);
    w.y = decltype(w.y)(widen(w.y) * sc);
    v.y[j][t] = w;
  }
}

// ---------------------------------------------------------------- Gram-Schmidt step in one launch
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// the double at this CTA's shared address p, in the CTA `rank` of the cluster
__device__ __forceinline__ double dsmem_ld(const double* p, unsigned rank) {
  unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(p)), b;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(b));
  return v;
}
template <class R>
__device__ __forceinline__ void cfma(R& cr, R& ci, R ar, R ai, R br, R bi) {
  cr = fma(ar, br, cr);
  cr = fma(-ai, bi, cr);
  ci = fma(ar, bi, ci);
  ci = fma(ai, br, ci);
}

// One cluster per right-hand side, its CTAs own slices of rows: classical
// Gram-Schmidt twice of column k + 1 against columns 0..k, its norm, the rotations
// and the scaling, with the partial sums exchanged through distributed shared
// memory.  For a small system the five launches of the separate kernels cost
// 10-13 us each whatever they do; the slices of the basis stay in L1 after the
// first of the four passes.
constexpr int GS_THREADS = 512, GS_WARPS = GS_THREADS / 32;
template <class CB, int CS>
__global__ void __launch_bounds__(GS_THREADS) gs_cluster_kernel(GivensArgs a, KrylovStep ks, int rs) {
  typedef typename Real<CB>::R R;
  extern __shared__ __align__(16) unsigned char gs_raw[];
  const int K = ks.k;  // columns 0 .. K - 1 against column K
  double2* hp = reinterpret_cast<double2*>(gs_raw);  // [2][K] this slice's sums
  double2* hd = hp + 2 * K;                          // [K + 1] both passes' coefficients added
  CB* hs = reinterpret_cast<CB*>(hd + K + 1);        // [K] in the arithmetic's precision
  CB* ws = hs + K + (K & 1);                         // [rs]
  CB* red = ws + rs;                                 // [GS_THREADS]
  Rot* rot = reinterpret_cast<Rot*>(red + GS_THREADS);  // [K], rank 0
  __shared__ double nred[GS_WARPS];
  __shared__ double npart, h1s, scs;
  const unsigned rank = cluster_rank();
  const int j = blockIdx.x / CS, r = a.on[j];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = int64_t(rank) * rs;
  const int rows = int(max(int64_t(0), min(int64_t(rs), ks.ldv - r0)));
  CB* V = reinterpret_cast<CB*>(ks.V[j]);
  CB* w = V + int64_t(K) * ks.ldv + r0;
  const bool live = a.st[r].live != 0;  // before the first cluster barrier: rank 0 changes it at the end
  for (int t = threadIdx.x; t < rows; t += GS_THREADS) ws[t] = w[t];
  if (rank == 0) stage_rotations(a, r, rot);
  __syncthreads();
  // update mapping: row tr of the slice, column group tg of ng
  const int rp = min(GS_THREADS, (rows + 31) / 32 * 32), ng = rp > 0 ? GS_THREADS / rp : 1;
  for (int pass = 0; pass < 2; ++pass) {
    double2* h = hp + pass * K;
    for (int i = warp; i < K; i += GS_WARPS) {
      const CB* v = V + int64_t(i) * ks.ldv + r0;
      R sr = 0, si = 0;
#pragma unroll 4
      for (int t = lane; t < rows; t += 32) {
        const CB x = v[t], y = ws[t];
        cfma(sr, si, x.x, -x.y, y.x, y.y);  // conj(v) w
      }
      const double dr = warp_total(widen(sr)), di = warp_total(widen(si));
      if (lane == 0) h[i] = make_double2(dr, di);
    }
    cluster_sync();
    for (int e = threadIdx.x; e < 2 * K; e += GS_THREADS) {
      double s = 0;
#pragma unroll
      for (int q = 0; q < CS; ++q) s += dsmem_ld(reinterpret_cast<const double*>(h) + e, q);
      reinterpret_cast<R*>(hs)[e] = R(s);
      double* o = reinterpret_cast<double*>(hd) + e;
      *o = pass ? *o + s : s;
    }
    __syncthreads();
    for (int tb = 0; tb < rows; tb += rp) {
      const int tr = tb + int(threadIdx.x) % rp, tg = int(threadIdx.x) / rp;
      R sr = 0, si = 0;
      if (tr < rows && tg < ng)
#pragma unroll 4
        for (int i = tg; i < K; i += ng) {
          const CB x = V[int64_t(i) * ks.ldv + r0 + tr], c = hs[i];
          cfma(sr, si, x.x, x.y, c.x, c.y);
        }
      red[threadIdx.x] = CB{sr, si};
      __syncthreads();
      if (tr < rows && tg == 0) {
        CB v = ws[tr];
        for (int q = 0; q < ng; ++q) {
          v.x -= red[q * rp + threadIdx.x].x;
          v.y -= red[q * rp + threadIdx.x].y;
        }
        ws[tr] = v;
      }
      __syncthreads();
    }
  }
  double nn = 0;
  for (int t = threadIdx.x; t < rows; t += GS_THREADS) {
    const double x = widen(ws[t].x), y = widen(ws[t].y);
    nn += x * x + y * y;
  }
  nn = warp_total(nn);
  if (lane == 0) nred[warp] = nn;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < GS_WARPS; ++q) nn += nred[q];
    npart = nn;
  }
  cluster_sync();
  if (warp == 0) {  // by one warp: FP64 instructions of the others would only queue behind it
    double total = lane < CS ? dsmem_ld(&npart, lane) : 0.0;
    total = warp_total(total);
    if (lane == 0) {
      h1s = sqrt(total);
      scs = live && total > 0 ? 1.0 / h1s : 0.0;
    }
  }
  __syncthreads();
  const double sc = scs;
  for (int t = threadIdx.x; t < rows; t += GS_THREADS) w[t] = cmake<CB>(widen(ws[t].x) * sc, widen(ws[t].y) * sc);
  if (rank == 0 && warp == 0) {
    if (live) givens_column(a, j, h1s, hd, rot);
    else if (lane == 0) a.flags[r] = 0;
  }
  cluster_sync();  // no CTA leaves while another may read its shared memory
}

// ---------------------------------------------------------------- end of a cycle
// one warp per right-hand side: back substitution, row by row from the bottom,
// the sum over the columns to the right split across the lanes
__global__ void gmres_backsolve_kernel(CycleEnd a) {
  const int r = a.on[blockIdx.x], m = a.m;
  const int ku = a.k[blockIdx.x];
  const double2* Hr = a.H + int64_t(r) * (m + 1) * m;
  const double2* gr = a.g + int64_t(r) * (m + 1);
  double2* y = a.dh + int64_t(r) * a.ldh;
  extern __shared__ __align__(16) unsigned char bs_raw[];
  double2* ys = reinterpret_cast<double2*>(bs_raw);
  const int lane = threadIdx.x;
  for (int i = ku - 1; i >= 0; --i) {
    double sr = 0, si = 0;
    const double2 d = Hr[int64_t(i) * m + i], gi = gr[i];
    for (int c = i + 1 + lane; c < ku; c += 32) {
      const double2 h = Hr[int64_t(i) * m + c], v = ys[c];
      sr += h.x * v.x - h.y * v.y;
      si += h.x * v.y + h.y * v.x;
    }
    sr = warp_total(sr);
    si = warp_total(si);
    if (lane == 0) {
      const double2 acc = make_double2(gi.x - sr, gi.y - si);
      const double dn = d.x * d.x + d.y * d.y;
      ys[i] = make_double2((acc.x * d.x + acc.y * d.y) / dn, (acc.y * d.x - acc.x * d.y) / dn);
    }
    __syncwarp();
  }
  for (int i = lane; i < ku; i += 32) y[i] = ys[i];
}

// out_j = V_j y_j in FP64.  A CTA owns 32 rows of one right-hand side; its 8 warps
// take every 8th Krylov column, four columns in flight, and the partial sums meet in
// shared memory.
template <class CB>
__global__ void __launch_bounds__(256) basis_sum_kernel(CycleEnd a, int64_t n) {
  __shared__ double part[8][32][2];
  const int j = blockIdx.y, k = a.k[j];
  const CB* __restrict__ V = reinterpret_cast<const CB*>(a.V[j]);
  const double2* __restrict__ h = a.dh + int64_t(a.on[j]) * a.ldh;
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int64_t t = int64_t(blockIdx.x) * 32 + lane;
  double sr = 0, si = 0;
  if (t < n) {
    int i = slice;
    for (; i + 24 < k; i += 32) {
      CB v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = V[int64_t(i + 8 * u) * a.ldv + t];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const double2 c = h[i + 8 * u];
        cfma(sr, si, widen(v[u].x), widen(v[u].y), c.x, c.y);
      }
    }
    for (; i < k; i += 8) {
      const CB v = V[int64_t(i) * a.ldv + t];
      const double2 c = h[i];
      cfma(sr, si, widen(v.x), widen(v.y), c.x, c.y);
    }
  }
  part[slice][lane][0] = sr;
  part[slice][lane][1] = si;
  __syncthreads();
  if (slice == 0 && t < n) {
    double ar = 0, ai = 0;
    for (int q = 0; q < 8; ++q) {
      ar += part[q][lane][0];
      ai += part[q][lane][1];
    }
    a.out[j][t] = make_double2(ar, ai);
  }
}

// x_j += diag(s1, 1, s3) w_j
__global__ void __launch_bounds__(256) add_scaled_kernel(int64_t n, int64_t ne, double s1, double s3, VecBatch<double2, double2> b) {
  const int64_t t = int64_t(blockIdx.x) * 256 + threadIdx.x;
  if (t >= n) return;
  const double s = t < ne ? s1 : (t < 2 * ne ? 1.0 : s3);
  const double2 w = b.x[blockIdx.y][t];
  double2& x = b.y[blockIdx.y][t];
  x = make_double2(fma(s, w.x, x.x), fma(s, w.y, x.y));
}

// ---------------------------------------------------------------- choice of the Gram-Schmidt form
// Cluster size: 8 is portable; complex128 steps, which the FP64 pipes of the
// cluster's SMs bound, take 16 where the device schedules them.
constexpr size_t GS_SMEM_MAX = 128 * 1024;
template <class CB, int CS>
bool launch_cluster(const GivensArgs& a, const KrylovStep& ks, cudaStream_t s) {
  const int rs = int((ks.ldv + CS * 32 - 1) / (CS * 32)) * 32;
  const size_t K = size_t(ks.k);
  const size_t smem = (3 * K + 1) * sizeof(double2) + (K + (K & 1) + rs + GS_THREADS) * sizeof(CB) + K * sizeof(Rot);
  int dev = 0;
  SLDM_CUDA(cudaGetDevice(&dev));
  static ClusterFit fit;
  if (smem > GS_SMEM_MAX || !cluster_fits(fit, dev, reinterpret_cast<const void*>(gs_cluster_kernel<CB, CS>), CS, GS_THREADS, GS_SMEM_MAX))
    return false;
  ClusterLaunch c(CS, unsigned(CS * ks.na), GS_THREADS, smem, s);
  SLDM_CUDA(cudaLaunchKernelEx(&c.cfg, gs_cluster_kernel<CB, CS>, a, ks, rs));
  count_launch();
  return true;
}

}  // namespace

void gmres_rhs(int64_t n, int64_t n2, double l, double2* b, double2* r, double* nrm, int nr, cudaStream_t s) {
  rhs_scale_kernel<<<dim3(unsigned((n + 255) / 256), nr), 256, 0, s>>>(n, n2, l, b, r, nrm), count_launch();
  SLDM_CUDA(cudaGetLastError());
}
void gmres_residual(int64_t n, const double2* b, const double2* y, double2* r, double* nrm, int nr, cudaStream_t s) {
  residual_kernel<<<dim3(unsigned((n + 255) / 256), nr), 256, 0, s>>>(n, b, y, r, nrm), count_launch();
  SLDM_CUDA(cudaGetLastError());
}
template <class CB>
void gmres_cycle_start(int64_t n, const CycleStart& a, int nr, cudaStream_t s) {
  cycle_start_kernel<CB><<<dim3(unsigned((n + 255) / 256), nr), 256, 0, s>>>(n, a), count_launch();
  SLDM_CUDA(cudaGetLastError());
}

// The one-launch step where its cluster's work is less than what the launches of the
// separate kernels cost: four passes over N (k + 1) entries per right-hand side.  Separate kernels
// against the cluster, us per step over a whole solve: complex128, N = 319 (28 steps) 41 / 25, 1,279 (40) 68 / 31, 5,119
// (54 steps, up to 2.8e5) 89 / 63; complex64, N = 1,279, 12 columns (51 steps) 38 / 21, 5,119 (69 steps, up to
// 3.5e5) 51 / 31, 8,631, 32 columns (up to 5e5 and more) 83 / 87.
constexpr double GS_MAX_C128 = 3.0e5, GS_MAX_C64 = 4.0e5;

template <class CB>
void gmres_orthogonalise(const GivensArgs& a, KrylovStep ks, double2* const* h1, double2* const* h2, cudaStream_t s) {
  const double work = double(ks.ldv) * ks.k;
  if (sizeof(CB) == sizeof(double2)) {
    if (work <= GS_MAX_C128 && (launch_cluster<CB, 16>(a, ks, s) || launch_cluster<CB, 8>(a, ks, s))) return;
  } else if (work <= GS_MAX_C64 && launch_cluster<CB, 8>(a, ks, s)) {
    return;
  }
  for (int j = 0; j < ks.na; ++j) ks.h[j] = h1[j];
  krylov_dots<CB>(ks, s);
  krylov_update<CB>(ks, false, s);
  for (int j = 0; j < ks.na; ++j) ks.h[j] = h2[j];
  krylov_dots<CB>(ks, s);
  krylov_update<CB>(ks, true, s);
  VecBatch<CB, CB> v;
  for (int j = 0; j < ks.na; ++j) v.y[j] = reinterpret_cast<CB*>(ks.V[j]) + int64_t(ks.k) * ks.ldv;
  const unsigned gx = unsigned(std::min<int64_t>((ks.n + 255) / 256, 1024));
  gmres_close_kernel<CB><<<dim3(gx + 1, ks.na), 256, size_t(ks.k + 1) * (sizeof(double2) + sizeof(Rot)), s>>>(a, v, ks.n),
      count_launch();
  SLDM_CUDA(cudaGetLastError());
}

template <class CB>
void gmres_cycle_end(int64_t n, const CycleEnd& a, int na, cudaStream_t s) {
  if (na <= 0) return;
  gmres_backsolve_kernel<<<na, 32, size_t(a.m) * sizeof(double2), s>>>(a), count_launch();
  basis_sum_kernel<CB><<<dim3(unsigned((n + 31) / 32), na), 256, 0, s>>>(a, n), count_launch();
  SLDM_CUDA(cudaGetLastError());
}
void gmres_add_scaled(int64_t n, int64_t ne, double s1, double s3, const VecBatch<double2, double2>& b, int na, cudaStream_t s) {
  add_scaled_kernel<<<dim3(unsigned((n + 255) / 256), na), 256, 0, s>>>(n, ne, s1, s3, b), count_launch();
  SLDM_CUDA(cudaGetLastError());
}

#define INST(C)                                                                                                        \
  template void gmres_cycle_start<C>(int64_t, const CycleStart&, int, cudaStream_t);                                  \
  template void gmres_orthogonalise<C>(const GivensArgs&, KrylovStep, double2* const*, double2* const*, cudaStream_t); \
  template void gmres_cycle_end<C>(int64_t, const CycleEnd&, int, cudaStream_t);
INST(float2)
INST(double2)
#undef INST

}  // namespace sldm
