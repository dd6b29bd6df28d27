// Backward Euler + Newton-Raphson for the 1D scheme (Sec. 5.1, Appendix A):
// one persistent thread-block cluster per instance runs time steps x Newton
// iterations (assembly, block cyclic reduction, update, convergence test).
// See include/dg_implicit.h.
#include <cmath>
#include <cstring>
#include <memory>
#include <string>
#include <vector>

#include "../../include/dg_implicit.h"
#include "dg_ctx.h"
#include "dg_kernels.cuh"

using namespace dgswe;

namespace {

template <int P, int M3>
struct IS {
  static constexpr int NP = P + 1, NE = M3 + 1, NB = 2 * NP + NE, NQ = (3 * P + 1) / 2;
};

template <int P, int M3>
struct ImplOps {
  using S = IS<P, M3>;
  double Vq[S::NQ * S::NP], dVq[S::NQ * S::NP];   // l_a, dl_a/dr at volume points
  double VEq[S::NQ * S::NE], dVEq[S::NQ * S::NE]; // psi_c, dpsi_c/dr
  double wq[S::NQ];
  double lf[2 * S::NP], lEf[2 * S::NE];           // basis at r = -1 (face 0) and r = +1 (face 1)
};

struct ImplArgs {
  int K;
  double dt, inv_dt, gc, gs, rho_inv, eta, sigma0, gamma, beta, pap_m, h_floor;
  int reg;
  double rtol, atol, xtol;
  int max_it, on_fail_continue;
  int n_gamma;    // > 1: continuation in gamma within each time step (Sec. 6.3)
  double gamma0;
  int mixed;  // 1: FP32 block factorization + FP64 iterative refinement
  BCEntry<double> bcL, bcR;
  double *X, *Uold, *R, *D, *L, *U, *Y, *DX;
  double *pt, *fc;               // pointwise data (volume_point, face_data)
  float *Df, *Lf, *Uf, *bf, *xf;  // mixed: FP32 copies of the system, its solution
  double* Rr;                    // mixed: refinement residual
  const double *J, *bed;
  double* red;  // reduction slots of the cluster
  dg_implicit_stats* st;
};

// sigma(E) and d sigma / dE in 1D (Eq. sigma11D, bingham1D regularized,
// Appendix A): sigma = (2 eta + phi(|E|)/(2|E|)) 2E, sigma' = 4 eta + phi'(|E|).
__device__ __forceinline__ void sigma1d(double e, const ImplArgs& a, double& sig, double& dsig) {
  Phys<double> ph{};
  ph.eta = a.eta;
  ph.sigma0 = a.sigma0;
  ph.gamma = a.gamma;
  ph.beta = a.beta;
  ph.half_inv_beta = 0.5 / a.beta;
  ph.pap_m = a.pap_m;
  ph.reg = a.reg;
  const double s = fabs(e);
  sig = (2.0 * a.eta + bingham_coef<double>(s, ph)) * 2.0 * e;
  double dp = 0.0;
  const double s0 = a.sigma0, g = a.gamma;
  if (a.reg != 0 && s0 != 0.0) {
    switch (a.reg) {
      case 1: {
        const double eps = 0.5 / a.beta, x = g * s - s0;
        const double mb = x >= eps ? x : (x <= -eps ? 0.0 : 0.5 * a.beta * (x + eps) * (x + eps));
        const double dmb = x >= eps ? 1.0 : (x <= -eps ? 0.0 : a.beta * (x + eps));
        const double den = mb + s0;
        dp = 2.0 * s0 * g / den - 2.0 * s0 * g * g * s * dmb / (den * den);
        break;
      }
      case 2: {
        const double eps = 0.5 / a.beta, x = g * s;
        dp = x >= s0 + eps ? 0.0 : (x <= s0 - eps ? 2.0 * g : 2.0 * a.beta * g * (s0 - x + eps));
        break;
      }
      case 3: {
        const double c = cosh(fmin(g * s, 350.0));
        dp = 2.0 * s0 * g / (c * c);
        break;
      }
      case 4: dp = 2.0 * s0 * a.pap_m * exp(-a.pap_m * s); break;
      case 5: dp = g * s < s0 ? 2.0 * g : 0.0; break;
    }
  }
  dsig = 4.0 * a.eta + dp;
}

__device__ __forceinline__ double block_sum(double v, double* sred) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sred[w] = v;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t += sred[i];
  return t;
}

// ------------------------------------------------------------------ thread-block cluster helpers
// The integrator runs on one cluster of thread blocks (up to eight SMs): a
// warp-wide FP64 instruction holds its sub-partition for 64 clocks however many
// of its lanes are active (measured 64-72), so the independent pieces of a
// Newton iteration are spread over the cluster's sub-partitions, and phases are
// separated by the cluster barrier (about 360 clocks, five FP64 instructions).
// 100 elements, p = 1, constant E, 3 Newton iterations a step: 2513 -> 265 us a
// step (one block with a one-warp block Thomas sweep before); FP32 elimination
// 1773 -> 330 us; p = 2, m3 = 2: 13.8 -> 1.1 ms; 400 elements: 33.3 -> 1.5 ms.

constexpr int kThreads = 256, kWarps = kThreads / 32, kMaxCluster = 8;

__device__ __forceinline__ int cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
// All threads of the cluster; orders their global-memory accesses.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Position of the thread in the cluster, and the reduction slots.
struct Team {
  int rank, size, tid, threads, warp, warps, lane;
  double* red;  // [4][kMaxCluster] global; slots used in turn
  int slot;
};

// Sum (MAX: maximum, NaNs skipped) over the cluster, the same value in every
// thread; blocks in rank order, so repeated runs agree.  Contains a cluster barrier.
template <bool MAX>
__device__ double team_reduce(double v, Team& t, double* sred) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double w = __shfl_down_sync(0xffffffffu, v, o);
    v = MAX ? fmax(v, w) : v + w;
  }
  __syncthreads();
  if (t.lane == 0) sred[threadIdx.x >> 5] = v;
  __syncthreads();
  double* slot = t.red + t.slot * kMaxCluster;
  if (threadIdx.x == 0) {
    double s = sred[0];
    for (int i = 1; i < kWarps; ++i) s = MAX ? fmax(s, sred[i]) : s + sred[i];
    slot[t.rank] = s;
  }
  cluster_sync();
  double s = slot[0];
  for (int i = 1; i < t.size; ++i) s = MAX ? fmax(s, slot[i]) : s + slot[i];
  t.slot = (t.slot + 1) & 3;
  return s;
}

// 1 / x of either sign
__device__ __forceinline__ double rcp_any(double x) {
  const double r = rcp_pos(fabs(x));
  return __hiloint2double(__double2hiint(r) | (__double2hiint(x) & (int)0x80000000u), __double2loint(r));
}
__device__ __forceinline__ float rcp_any(float x) { return 1.0f / x; }

// ------------------------------------------------------------------ assembly

// Pointwise data of a Newton iterate, one item per thread (kPt doubles a volume
// point, kFc a face): every face is evaluated once.
constexpr int kPt = 5;   // h, u, sigma, sigma', dH/dx
constexpr int kFc = 17;  // F_h, F_u, G; d(F_h, F_u)/d(h, u) left and right; dF_u/dE left, right; dG/du left, right

template <int P, int M3>
__device__ void volume_point(int i, const ImplArgs& a, const ImplOps<P, M3>& o) {
  using S = IS<P, M3>;
  constexpr int NP = S::NP, NE = S::NE, NB = S::NB, NQ = S::NQ;
  const int e = i / NQ, q = i - e * NQ;
  const double* x = a.X + (size_t)e * NB;
  double h = 0, u = 0, ee = 0, dH = 0;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    h += o.Vq[q * NP + k] * x[k];
    u += o.Vq[q * NP + k] * x[NP + k];
    if (a.bed) dH += o.dVq[q * NP + k] * a.bed[(size_t)e * NP + k];
  }
#pragma unroll
  for (int c = 0; c < NE; ++c) ee += o.VEq[q * NE + c] * x[2 * NP + c];
  double* p = a.pt + (size_t)i * kPt;
  p[0] = h;
  p[1] = u;
  sigma1d(ee, a, p[2], p[3]);
  p[4] = a.bed ? dH / a.J[e] : 0.0;
}

// Face i between elements i - 1 and i, normal +1: numerical flux F (HLL minus
// the central flux of Q), central G, and their derivatives with the HLL speeds
// held fixed.  At the ends the missing side is the ghost state, its derivatives
// taken through the ghost's dependence on the inner state.
template <int P, int M3>
__device__ void face_data(int i, const ImplArgs& a, const ImplOps<P, M3>& o) {
  using S = IS<P, M3>;
  constexpr int NP = S::NP, NE = S::NE, NB = S::NB;
  double h[2], u[2], ee[2];                          // left, right
  double dh[2] = {1, 1}, du[2] = {1, 1}, de[2] = {1, 1};  // d ghost / d inner
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int e = i - 1 + s, f = 1 - s;  // the left element's face 1, the right one's face 0
    h[s] = u[s] = ee[s] = 0.0;
    if (e >= 0 && e < a.K) {
      const double* x = a.X + (size_t)e * NB;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        h[s] += o.lf[f * NP + k] * x[k];
        u[s] += o.lf[f * NP + k] * x[NP + k];
      }
#pragma unroll
      for (int c = 0; c < NE; ++c) ee[s] += o.lEf[f * NE + c] * x[2 * NP + c];
    }
  }
  if (i == 0 || i == a.K) {
    const int g = i == 0 ? 0 : 1, in = 1 - g;  // ghost side, inner side
    const BCEntry<double>& b = i == 0 ? a.bcL : a.bcR;
    const bool d0 = b.mode[0] == 1, d1 = b.mode[1] == 1, w = b.mode[1] == 2, d2 = b.mode[2] == 1;
    const double gh = d0 ? b.val[0] : h[in], gu = d1 ? b.val[1] : w ? -u[in] : u[in], ge = d2 ? b.val[2] : ee[in];
    const double fh = d0 ? 0.0 : 1.0, fu = d1 ? 0.0 : w ? -1.0 : 1.0, fe = d2 ? 0.0 : 1.0;
    if (g == 0) {
      h[0] = gh, u[0] = gu, ee[0] = ge, dh[0] = fh, du[0] = fu, de[0] = fe;
    } else {
      h[1] = gh, u[1] = gu, ee[1] = ge, dh[1] = fh, du[1] = fu, de[1] = fe;
    }
  }
  double c[2], F0[2], F1[2], sg[2], ds[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    c[s] = sqrt_pos(a.gc * fmax(h[s], a.h_floor));
    F0[s] = h[s] * u[s];
    F1[s] = F0[s] * u[s] + (0.5 * a.gc) * h[s] * h[s];
    sigma1d(ee[s], a, sg[s], ds[s]);
  }
  const double SL = fmin(u[0] - c[0], u[1] - c[1]), SR = fmax(u[0] + c[0], u[1] + c[1]);
  // F = x F_left + y F_right + z (U_right - U_left)
  double x = 1.0, y = 0.0, z = 0.0;
  if (SL >= 0.0) {
  } else if (SR <= 0.0) {
    x = 0.0;
    y = 1.0;
  } else {
    const double inv = rcp_pos(SR - SL);
    x = SR * inv;
    y = -SL * inv;
    z = SL * x;
  }
  double* p = a.fc + (size_t)i * kFc;
  const double hr = 0.5 * a.rho_inv;
  p[0] = x * F0[0] + (y * F0[1] + z * (h[1] - h[0]));
  p[1] = x * F1[0] + (y * F1[1] + z * (F0[1] - F0[0])) - hr * (h[0] * sg[0] + h[1] * sg[1]);
  p[2] = 0.5 * (u[0] + u[1]);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double wf = s == 0 ? x : y, wu = s == 0 ? -z : z;  // weights of dF and dU of the side
    double* A = p + 3 + 4 * s;
    A[0] = (wf * u[s] + wu) * dh[s];
    A[1] = (wf * h[s]) * du[s];
    A[2] = (wf * (u[s] * u[s] + a.gc * h[s]) + wu * u[s] - hr * sg[s]) * dh[s];
    A[3] = (wf * (2.0 * h[s] * u[s]) + wu * h[s]) * du[s];
    p[11 + s] = -hr * h[s] * ds[s] * de[s];
    p[13 + s] = 0.5 * du[s];
  }
}

// Row r of element e: residual entry and the rows of the blocks D (own), L (left
// neighbour), U (right neighbour).  Returns the residual entry.
template <int P, int M3>
__device__ double assemble_row(int e, int r, const ImplArgs& a, const ImplOps<P, M3>& o) {
  using S = IS<P, M3>;
  constexpr int NP = S::NP, NE = S::NE, NB = S::NB, NQ = S::NQ;
  const double J = a.J[e];
  const int rb = r < NP ? 0 : (r < 2 * NP ? 1 : 2);  // row block: h, u, E
  const int ri = rb < 2 ? r - rb * NP : r - 2 * NP;
  double res = rb < 2 ? -a.Uold[(size_t)e * 2 * NP + r] * a.inv_dt : 0.0;
  double D[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) D[c] = 0.0;
#pragma unroll
  for (int q = 0; q < NQ; ++q) {
    const double* p = a.pt + ((size_t)e * NQ + q) * kPt;
    const double h = p[0], u = p[1], w = o.wq[q];
    const double m = w * J * (rb < 2 ? o.Vq[q * NP + ri] : o.VEq[q * NE + ri]);
    const double d = w * (rb < 2 ? o.dVq[q * NP + ri] : o.dVEq[q * NE + ri]);
    double ch = 0.0, cu = 0.0, ce = 0.0;
    if (rb == 0) {
      const double mt = m * a.inv_dt;
      ch = mt - d * u;
      cu = -d * h;
      res += ch * h;
    } else if (rb == 1) {
      const double mt = m * a.inv_dt, s = p[2] * a.rho_inv, f = a.gs + a.gc * p[4], hu = h * u;
      ch = mt * u + d * (s - (u * u + a.gc * h)) + m * f;
      cu = mt * h - 2.0 * d * hu;
      ce = d * (h * p[3] * a.rho_inv);
      res += mt * hu + d * (h * s - (hu * u + 0.5 * a.gc * h * h)) + m * f * h;
    } else {
      cu = d;
      ce = m;
      double ee = 0.0;
#pragma unroll
      for (int c = 0; c < NE; ++c) ee += o.VEq[q * NE + c] * a.X[(size_t)e * NB + 2 * NP + c];
      res += m * ee + d * u;
    }
#pragma unroll
    for (int c = 0; c < NP; ++c) {
      D[c] += ch * o.Vq[q * NP + c];
      D[NP + c] += cu * o.Vq[q * NP + c];
    }
#pragma unroll
    for (int c = 0; c < NE; ++c) D[2 * NP + c] += ce * o.VEq[q * NE + c];
  }
  // faces: 0 (left, the face data's right side is own) and 1
  double* Dm = a.D + ((size_t)e * NB + r) * NB;
  double* Lm = a.L + ((size_t)e * NB + r) * NB;
  double* Um = a.U + ((size_t)e * NB + r) * NB;
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const double* p = a.fc + (size_t)(e + f) * kFc;
    const double fr = (f == 0 ? -1.0 : 1.0) * (rb < 2 ? o.lf[f * NP + ri] : o.lEf[f * NE + ri]);
    const int own = 1 - f, out = f;  // side of the own and of the outer state
    double vo[3] = {0, 0, 0}, vx[3] = {0, 0, 0};  // d/d(h, u, E) of the own and the outer trace
    if (rb < 2) {
      res += fr * p[rb];
      vo[0] = fr * p[3 + 4 * own + 2 * rb];
      vo[1] = fr * p[3 + 4 * own + 2 * rb + 1];
      vx[0] = fr * p[3 + 4 * out + 2 * rb];
      vx[1] = fr * p[3 + 4 * out + 2 * rb + 1];
      if (rb == 1) {
        vo[2] = fr * p[11 + own];
        vx[2] = fr * p[11 + out];
      }
    } else {
      res -= fr * p[2];
      vo[1] = -fr * p[13 + own];
      vx[1] = -fr * p[13 + out];
    }
    const bool end = f == 0 ? e == 0 : e == a.K - 1;  // the outer state is the ghost of the own one
    double* N = f == 0 ? Lm : Um;
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int cb = c < NP ? 0 : (c < 2 * NP ? 1 : 2);
      const int ci = cb < 2 ? c - cb * NP : c - 2 * NP;
      const double lo = cb < 2 ? o.lf[f * NP + ci] : o.lEf[f * NE + ci];
      const double lx = cb < 2 ? o.lf[(1 - f) * NP + ci] : o.lEf[(1 - f) * NE + ci];
      D[c] += (end ? vo[cb] + vx[cb] : vo[cb]) * lo;
      N[c] = end ? 0.0 : vx[cb] * lx;
    }
  }
#pragma unroll
  for (int c = 0; c < NB; ++c) Dm[c] = D[c];
  a.R[(size_t)e * NB + r] = res;
  return res;
}

// ------------------------------------------------------------------ block cyclic reduction

// Block-tridiagonal system in T: blocks D, L, U [K][NB][NB] and right-hand side
// b [K][NB], overwritten; solution x.  Cyclic reduction: at stride s the rows
// i = s - 1, 3 s - 1, .. of those left are eliminated (P = D^-1 L, Q = D^-1 U,
// r = D^-1 b replace L, U, b) and the rows between them updated, so a solve is
// log2 K elimination steps deep instead of K; a row's elimination is a
// Gauss-Jordan with partial pivoting of [D | L | U | b] by one warp, a column
// per lane (two per lane beyond 32 columns).
template <typename T>
struct BTri {
  T *D, *L, *U, *b;
  int K;
};

template <typename T, int NB>
struct BCols {
  static constexpr int N = 3 * NB + 1, NC = (N + 31) / 32;
};

// Gauss-Jordan of the warp's columns; columns 0 .. NB - 1 become the identity.
template <typename T, int NB>
__device__ __forceinline__ void gauss_jordan(T (&col)[BCols<T, NB>::NC][NB]) {
  constexpr int NC = BCols<T, NB>::NC;
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    int piv = k;
    T best = fabs(col[0][k]);
#pragma unroll
    for (int r = k + 1; r < NB; ++r) {
      const T v = fabs(col[0][r]);
      if (less_pos<T>(best, v)) {
        best = v;
        piv = r;
      }
    }
    piv = __shfl_sync(0xffffffffu, piv, k);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
#pragma unroll
      for (int r = k + 1; r < NB; ++r)
        if (r == piv) {
          const T t = col[c][k];
          col[c][k] = col[c][r];
          col[c][r] = t;
        }
    }
    T f[NB];
#pragma unroll
    for (int r = 0; r < NB; ++r) f[r] = __shfl_sync(0xffffffffu, col[0][r], k);
    const T inv = rcp_any(f[k]);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      col[c][k] *= inv;
#pragma unroll
      for (int r = 0; r < NB; ++r)
        if (r != k) col[c][r] -= f[r] * col[c][k];
    }
  }
}

// Row i: update by its eliminated neighbours i - s, i + s (s = 0: none), then,
// if elim, elimination.
template <typename T, int NB>
__device__ void bcr_row(const BTri<T>& A, int i, int s, bool elim, int lane) {
  constexpr int NC = BCols<T, NB>::NC, B2 = NB * NB;
  const int lft = i - s, rgt = i + s;
  const bool hr = s > 0 && rgt < A.K;
  T col[NC][NB];
  T* Di = A.D + (size_t)i * B2;
  T* Li = A.L + (size_t)i * B2;
  T* Ui = A.U + (size_t)i * B2;
#pragma unroll
  for (int cc = 0; cc < NC; ++cc) {
    const int c = lane + 32 * cc, kind = c < NB ? 0 : c < 2 * NB ? 1 : c < 3 * NB ? 2 : 3, j = c - kind * NB;
    const bool in = c < 3 * NB + 1;
    // base column, and the neighbours' columns that L_i and U_i multiply
    const T* base = kind == 0 ? Di + j : kind == 1 ? Li + j : kind == 2 ? Ui + j : A.b + (size_t)i * NB;
    const int st = kind == 3 ? 1 : NB;
    const bool keep = s == 0 || kind == 0 || kind == 3;
#pragma unroll
    for (int r = 0; r < NB; ++r) col[cc][r] = in && keep ? base[r * st] : T(0);
    if (s > 0) {
      T v[NB], w[NB];
      const T* vp = kind == 0 ? A.U + (size_t)lft * B2 + j : kind == 1 ? A.L + (size_t)lft * B2 + j : A.b + (size_t)lft * NB;
      const T* wp = kind == 0 ? A.L + (size_t)rgt * B2 + j : kind == 2 ? A.U + (size_t)rgt * B2 + j : A.b + (size_t)rgt * NB;
      const bool hv = in && kind != 2, hw = in && hr && kind != 1;
#pragma unroll
      for (int m = 0; m < NB; ++m) {
        v[m] = hv ? vp[m * st] : T(0);
        w[m] = hw ? wp[m * st] : T(0);
      }
#pragma unroll
      for (int r = 0; r < NB; ++r) {
        T t = col[cc][r];
#pragma unroll
        for (int m = 0; m < NB; ++m) t -= Li[r * NB + m] * v[m];
        if (hr) {
#pragma unroll
          for (int m = 0; m < NB; ++m) t -= Ui[r * NB + m] * w[m];
        }
        col[cc][r] = t;
      }
    }
  }
  __syncwarp();  // every lane has read the row's blocks
  if (elim) gauss_jordan<T, NB>(col);
#pragma unroll
  for (int cc = 0; cc < NC; ++cc) {
    const int c = lane + 32 * cc, kind = c < NB ? 0 : c < 2 * NB ? 1 : c < 3 * NB ? 2 : 3, j = c - kind * NB;
    if (c >= 3 * NB + 1 || (elim && kind == 0)) continue;
    T* dst = kind == 0 ? Di + j : kind == 1 ? Li + j : kind == 2 ? Ui + j : A.b + (size_t)i * NB;
    const int st = kind == 3 ? 1 : NB;
#pragma unroll
    for (int r = 0; r < NB; ++r) dst[r * st] = col[cc][r];
  }
}

// x of the system; all threads of the cluster (blocks, b written and ordered
// before the call; x is ordered for all threads after it).
template <typename T, int NB>
__device__ void bcr_solve(const BTri<T>& A, T* x, const Team& t) {
  const int K = A.K;
  // stride s: the rows left are s - 1, 2 s - 1, ..; n of them.  A row left at
  // stride s was updated by those eliminated at s / 2.
  int s = 1;
  for (;; s *= 2) {
    const int n = K / s;
    for (int k = t.warp; k < n; k += t.warps)
      if ((k & 1) == 0 || s > 1) bcr_row<T, NB>(A, (k + 1) * s - 1, s / 2, (k & 1) == 0, t.lane);
    cluster_sync();
    if (n <= 1) break;
  }
  // back: rows eliminated at stride s, whose neighbours at distance s are known
  for (; s >= 1; s /= 2) {
    const int n = (K / s + 1) / 2 * NB;  // eliminated rows times unknowns
    for (int k = t.tid; k < n; k += t.threads) {
      const int i = (2 * (k / NB) + 1) * s - 1, r = k % NB;
      T v = A.b[(size_t)i * NB + r];
      const T* Pm = A.L + ((size_t)i * NB + r) * NB;
      const T* Qm = A.U + ((size_t)i * NB + r) * NB;
      if (i - s >= 0) {
#pragma unroll
        for (int m = 0; m < NB; ++m) v -= Pm[m] * x[(size_t)(i - s) * NB + m];
      }
      if (i + s < K) {
#pragma unroll
        for (int m = 0; m < NB; ++m) v -= Qm[m] * x[(size_t)(i + s) * NB + m];
      }
      x[(size_t)i * NB + r] = v;
    }
    cluster_sync();
  }
}

// FP64 residual of the linear system, r = -R - J dx (block tridiagonal).
template <int NB>
__device__ void linear_residual_f64(const ImplArgs& a, const Team& t) {
  for (int i = t.tid; i < a.K * NB; i += t.threads) {
    const int e = i / NB, r = i - e * NB;
    double v = -a.R[i];
    const double* D = a.D + (size_t)e * NB * NB + (size_t)r * NB;
    const double* x = a.DX + (size_t)e * NB;
#pragma unroll
    for (int j = 0; j < NB; ++j) v -= D[j] * x[j];
    if (e > 0) {
      const double* L = a.L + (size_t)e * NB * NB + (size_t)r * NB;
#pragma unroll
      for (int j = 0; j < NB; ++j) v -= L[j] * x[j - NB];
    }
    if (e < a.K - 1) {
      const double* U = a.U + (size_t)e * NB * NB + (size_t)r * NB;
#pragma unroll
      for (int j = 0; j < NB; ++j) v -= U[j] * x[j + NB];
    }
    a.Rr[i] = v;
  }
}

// FP32 block factorization and solve of J x = b (b in FP64), on float copies of
// the blocks.
template <int NB>
__device__ void solve_f32(const ImplArgs& a, const double* b, float* x, const Team& t) {
  const BTri<float> A{a.Df, a.Lf, a.Uf, a.bf, a.K};
  const size_t nb = (size_t)a.K * NB, n = nb * NB;  // the blocks' entries can pass 2^31
  for (size_t i = t.tid; i < n; i += t.threads) {
    a.Df[i] = (float)a.D[i];
    a.Lf[i] = (float)a.L[i];
    a.Uf[i] = (float)a.U[i];
    if (i < nb) a.bf[i] = (float)b[i];
  }
  cluster_sync();
  bcr_solve<float, NB>(A, x, t);
}

constexpr int kRefinements = 2;

// Newton iteration for one time level (and one continuation stage): returns
// the iteration count, whether it converged and max |x|.
template <int P, int M3>
__device__ void newton_solve(const ImplArgs& a, const ImplOps<P, M3>& o, Team& t, double* sred, int& its_out,
                             bool& conv_out, double& xmax_out) {
  using S = IS<P, M3>;
  constexpr int NB = S::NB, NQ = S::NQ;
  const int K = a.K;
  double r0 = 0.0, dxmax = 0.0, xmax = 0.0;
  int its = 0;
  bool conv = false;
  for (int it = 0;; ++it) {
    // faces first (the longer items), volume points after them
    for (int i = t.tid; i < K + 1 + K * NQ; i += t.threads) {
      if (i <= K) face_data<P, M3>(i, a, o);
      else volume_point<P, M3>(i - K - 1, a, o);
    }
    cluster_sync();
    double part = 0.0;
    for (int i = t.tid; i < K * NB; i += t.threads) {
      const int r = i / K, e = i - r * K;  // a warp's rows are of one kind
      const double v = assemble_row<P, M3>(e, r, a, o);
      part += v * v;
      (a.mixed ? a.Rr : a.Y)[(size_t)e * NB + r] = -v;
    }
    const double rn = sqrt(team_reduce<false>(part, t, sred));
    if (it == 0) {
      r0 = rn;
      if (rn <= a.atol) {
        conv = true;
        its = 0;
        break;
      }
    } else if (rn <= a.rtol * r0 || rn <= a.atol || dxmax <= a.xtol * (1.0 + xmax)) {
      conv = true;
      its = it;
      break;
    }
    if (it == a.max_it || !(rn == rn)) {
      its = it;
      break;
    }
    double dm = 0.0, xm = 0.0;
    if (a.mixed) {
      // FP32 factorization and solve, then rounds of FP64 residual and FP32 correction
      solve_f32<NB>(a, a.Rr, a.xf, t);
      for (int i = t.tid; i < K * NB; i += t.threads) a.DX[i] = (double)a.xf[i];
      cluster_sync();
      for (int ref = 0; ref < kRefinements; ++ref) {
        linear_residual_f64<NB>(a, t);
        cluster_sync();
        solve_f32<NB>(a, a.Rr, a.xf, t);
        for (int i = t.tid; i < K * NB; i += t.threads) a.DX[i] += (double)a.xf[i];
        cluster_sync();
      }
    } else {
      bcr_solve<double, NB>(BTri<double>{a.D, a.L, a.U, a.Y, K}, a.DX, t);
    }
    for (int i = t.tid; i < K * NB; i += t.threads) {
      const double d = a.DX[i];
      const double xn = a.X[i] + d;
      a.X[i] = xn;
      dm = fmax(dm, fabs(d));
      xm = fmax(xm, fabs(xn));
    }
    dxmax = team_reduce<true>(dm, t, sred);
    xmax = team_reduce<true>(xm, t, sred);
  }
  its_out = its;
  conv_out = conv;
  xmax_out = xmax;
}

template <int P, int M3>
__global__ void __launch_bounds__(kThreads) implicit_kernel(ImplArgs a, ImplOps<P, M3> o, long long n_steps) {
  using S = IS<P, M3>;
  constexpr int NP = S::NP, NB = S::NB, NQ = S::NQ;
  __shared__ double sred[kWarps];
  const int K = a.K;
  Team t;
  t.rank = cluster_rank();
  t.size = cluster_size();
  // consecutive warps of items go to different blocks, then to different sub-partitions
  t.lane = threadIdx.x & 31;
  t.warp = (threadIdx.x >> 5) * t.size + t.rank;
  t.warps = kWarps * t.size;
  t.tid = t.warp * 32 + t.lane;
  t.threads = t.warps * 32;
  t.red = a.red;
  t.slot = 0;
  for (long long step = 0; step < n_steps; ++step) {
    // <N_V, U(V^{k-1})>
    for (int i = t.tid; i < K * NP; i += t.threads) {
      const int e = i / NP, k = i - e * NP;
      const double* x = a.X + (size_t)e * NB;
      const double J = a.J[e];
      double s0 = 0, s1 = 0;
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        double hh = 0, uu = 0;
#pragma unroll
        for (int j = 0; j < NP; ++j) {
          hh += o.Vq[q * NP + j] * x[j];
          uu += o.Vq[q * NP + j] * x[NP + j];
        }
        const double w = o.wq[q] * J * o.Vq[q * NP + k];
        s0 += w * hh;
        s1 += w * (hh * uu);
      }
      a.Uold[(size_t)e * 2 * NP + k] = s0;
      a.Uold[(size_t)e * 2 * NP + NP + k] = s1;
    }
    // (Uold is read after the first barrier of newton_solve)
    // continuation in gamma (Sec. 6.3): gamma_i = gamma0 + (i-1)(gamma-gamma0)/(n_gamma-1)
    const int ng = a.n_gamma > 1 ? a.n_gamma : 1;
    int its = 0;
    bool conv = true;
    double xmax = 0.0;
    for (int ic = 0; ic < ng; ++ic) {
      ImplArgs b = a;
      if (ng > 1) b.gamma = a.gamma0 + ic * (a.gamma - a.gamma0) / (ng - 1);
      int it_s;
      bool cv_s;
      newton_solve<P, M3>(b, o, t, sred, it_s, cv_s, xmax);
      its += it_s;
      conv = conv && cv_s;
    }
    if (t.tid == 0) {
      dg_implicit_stats& st = *a.st;
      st.steps += 1;
      st.t += a.dt;
      st.newton_its += its;
      st.last_its = its;
      if (!conv) st.failed_steps += 1;
      if (!(xmax == xmax)) st.status = DG_ERR_NONFINITE;
      else if (!conv && !a.on_fail_continue) st.status = DG_ERR_NEWTON;
    }
    cluster_sync();
    if (a.st->status != 0) break;
  }
}

// E consistent with V (R_E = 0; element-local solve of <N_E, N_E> E = rhs),
// thread per element.  Also the active-region indicator per element.
template <int P, int M3>
__global__ void init_E_kernel(ImplArgs a, ImplOps<P, M3> o, const double* __restrict__ MEinv) {
  using S = IS<P, M3>;
  constexpr int NP = S::NP, NE = S::NE, NB = S::NB, NQ = S::NQ;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.K) return;
  double* x = a.X + (size_t)e * NB;
  const double J = a.J[e];
  double rhs[NE];
#pragma unroll
  for (int c = 0; c < NE; ++c) {
    double r = 0.0;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      double uu = 0.0;
#pragma unroll
      for (int j = 0; j < NP; ++j) uu += o.Vq[q * NP + j] * x[NP + j];
      r -= o.wq[q] * o.dVEq[q * NE + c] * uu;
    }
    rhs[c] = r;
  }
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const double n = f == 0 ? -1.0 : 1.0;
    double um = 0.0;
#pragma unroll
    for (int j = 0; j < NP; ++j) um += o.lf[f * NP + j] * x[NP + j];
    double up;
    const int e2 = f == 0 ? e - 1 : e + 1;
    if (e2 >= 0 && e2 < a.K) {
      up = 0.0;
#pragma unroll
      for (int j = 0; j < NP; ++j) up += o.lf[(1 - f) * NP + j] * a.X[(size_t)e2 * NB + NP + j];
    } else {
      const BCEntry<double>& b = f == 0 ? a.bcL : a.bcR;
      up = b.mode[1] == 1 ? b.val[1] : (b.mode[1] == 2 ? -um : um);
    }
#pragma unroll
    for (int c = 0; c < NE; ++c) rhs[c] += o.lEf[f * NE + c] * 0.5 * (um + up) * n;
  }
  // written to a scratch row first: neighbours read this element's u only
#pragma unroll
  for (int c = 0; c < NE; ++c) {
    double v = 0.0;
#pragma unroll
    for (int d = 0; d < NE; ++d) v += MEinv[c * NE + d] * rhs[d];
    a.DX[(size_t)e * NB + c] = v / J;
  }
}

template <int P, int M3>
__global__ void commit_E_kernel(ImplArgs a) {
  using S = IS<P, M3>;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= a.K) return;
#pragma unroll
  for (int c = 0; c < S::NE; ++c) a.X[(size_t)e * S::NB + 2 * S::NP + c] = a.DX[(size_t)e * S::NB + c];
}

template <int P, int M3>
__global__ void active_kernel(ImplArgs a, ImplOps<P, M3> o, double* out) {
  using S = IS<P, M3>;
  constexpr int NE = S::NE, NB = S::NB, NQ = S::NQ;
  __shared__ double sred[32];
  double act = 0.0, tot = 0.0;
  const double thr = a.gamma > 0 ? a.sigma0 / a.gamma : 0.0;
  for (int e = threadIdx.x; e < a.K; e += blockDim.x) {
    const double* x = a.X + (size_t)e * NB + 2 * S::NP;
    for (int q = 0; q < NQ; ++q) {
      double ee = 0.0;
      for (int c = 0; c < NE; ++c) ee += o.VEq[q * NE + c] * x[c];
      const double w = o.wq[q] * a.J[e];
      tot += w;
      if (fabs(ee) - thr >= 0.0) act += w;
    }
  }
  const double A = block_sum(act, sred);
  const double T = block_sum(tot, sred);
  if (threadIdx.x == 0) *out = 100.0 * A / T;
}

struct ImplDrv {
  virtual ~ImplDrv() = default;
  virtual void run(dg_implicit* s, long long n, cudaStream_t st) = 0;
  virtual void init_E(dg_implicit* s, cudaStream_t st) = 0;
  virtual void active(dg_implicit* s, double* out, cudaStream_t st) = 0;
};

}  // namespace

struct dg_implicit {
  int p = 0, m3 = 0, reg = 0;
  int64_t K = 0;
  dg_swe_params prm{};
  dg_implicit_params ip{};
  std::vector<double> J, bed, node_x, MEinv;
  std::vector<double> Vq, dVq, VEq, dVEq, wq, lf, lEf;
  BCEntry<double> bcL{}, bcR{};
  bool has_bed = false;
  size_t ws_need = 0;
  char* ws = nullptr;
  struct {
    size_t X, Uold, R, D, L, U, Y, DX, J, bed, red, st, MEinv, act, pt, fc, Df, Lf, Uf, bf, xf, Rr;
  } off{};
  cudaStream_t stream = nullptr;
  std::unique_ptr<ImplDrv> drv;
  std::string err;
  template <typename T>
  T* at(size_t o) const { return reinterpret_cast<T*>(ws + o); }
  int nb() const { return 2 * (p + 1) + (m3 + 1); }
};

namespace {

dg_status ifail(dg_implicit* s, dg_status st, const std::string& m) {
  if (s) s->err = m;
  return st;
}
#define IK(call)                                                                     \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) return ifail(s, DG_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

ImplArgs make_args(dg_implicit* s) {
  ImplArgs a{};
  const auto& p = s->prm;
  a.K = (int)s->K;
  a.dt = s->ip.dt;
  a.inv_dt = 1.0 / s->ip.dt;
  a.gc = p.g * std::cos(p.alpha);
  a.gs = p.g * std::sin(p.alpha);
  a.rho_inv = 1.0 / p.rho;
  a.eta = p.eta;
  a.sigma0 = p.sigma0;
  a.gamma = p.gamma;
  a.beta = p.beta;
  a.pap_m = p.pap_m;
  a.h_floor = p.h_floor;
  a.reg = s->reg;
  a.rtol = s->ip.rtol;
  a.atol = s->ip.atol;
  a.xtol = s->ip.xtol;
  a.max_it = s->ip.max_it;
  a.on_fail_continue = s->ip.on_fail_continue;
  a.mixed = s->ip.linear_solver == 1 ? 1 : 0;
  a.n_gamma = s->ip.n_gamma;
  a.gamma0 = s->ip.gamma0;
  a.Df = s->at<float>(s->off.Df);
  a.Lf = s->at<float>(s->off.Lf);
  a.Uf = s->at<float>(s->off.Uf);
  a.bf = s->at<float>(s->off.bf);
  a.xf = s->at<float>(s->off.xf);
  a.Rr = s->at<double>(s->off.Rr);
  a.pt = s->at<double>(s->off.pt);
  a.fc = s->at<double>(s->off.fc);
  a.bcL = s->bcL;
  a.bcR = s->bcR;
  a.X = s->at<double>(s->off.X);
  a.Uold = s->at<double>(s->off.Uold);
  a.R = s->at<double>(s->off.R);
  a.D = s->at<double>(s->off.D);
  a.L = s->at<double>(s->off.L);
  a.U = s->at<double>(s->off.U);
  a.Y = s->at<double>(s->off.Y);
  a.DX = s->at<double>(s->off.DX);
  a.J = s->at<double>(s->off.J);
  a.bed = s->has_bed ? s->at<double>(s->off.bed) : nullptr;
  a.red = s->at<double>(s->off.red);
  a.st = s->at<dg_implicit_stats>(s->off.st);
  return a;
}

template <int P, int M3>
struct IDrv final : ImplDrv {
  ImplOps<P, M3> o{};
  explicit IDrv(const dg_implicit& s) {
    using S = IS<P, M3>;
    for (int i = 0; i < S::NQ * S::NP; ++i) {
      o.Vq[i] = s.Vq[i];
      o.dVq[i] = s.dVq[i];
    }
    for (int i = 0; i < S::NQ * S::NE; ++i) {
      o.VEq[i] = s.VEq[i];
      o.dVEq[i] = s.dVEq[i];
    }
    for (int q = 0; q < S::NQ; ++q) o.wq[q] = s.wq[q];
    for (int i = 0; i < 2 * S::NP; ++i) o.lf[i] = s.lf[i];
    for (int i = 0; i < 2 * S::NE; ++i) o.lEf[i] = s.lEf[i];
  }
  void run(dg_implicit* s, long long n, cudaStream_t st) override {
    // one cluster: eight blocks from 12 elements on, where the phases have work
    // for several warps; below, one block and its cheaper barrier
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = s->K >= 12 ? kMaxCluster : 1;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(at.val.clusterDim.x);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, implicit_kernel<P, M3>, make_args(s), o, n);
  }
  void init_E(dg_implicit* s, cudaStream_t st) override {
    const int K = (int)s->K;
    init_E_kernel<P, M3><<<(K + 127) / 128, 128, 0, st>>>(make_args(s), o, s->at<double>(s->off.MEinv));
    commit_E_kernel<P, M3><<<(K + 127) / 128, 128, 0, st>>>(make_args(s));
  }
  void active(dg_implicit* s, double* out, cudaStream_t st) override {
    active_kernel<P, M3><<<1, 256, 0, st>>>(make_args(s), o, out);
  }
};

std::unique_ptr<ImplDrv> make_idrv(const dg_implicit& s) {
#define ICASE(PP, MM) \
  if (s.p == PP && s.m3 == MM) return std::unique_ptr<ImplDrv>(new IDrv<PP, MM>(s));
  ICASE(1, 0) ICASE(1, 1) ICASE(2, 0) ICASE(2, 1) ICASE(2, 2) ICASE(3, 0) ICASE(3, 1) ICASE(3, 2) ICASE(3, 3)
#undef ICASE
  return nullptr;
}

// 1D Lagrange basis on equispaced nodes of degree m (m = 0: the constant 1).
void lagrange1d(int m, double r, double* l, double* dl) {
  if (m == 0) {
    l[0] = 1.0;
    dl[0] = 0.0;
    return;
  }
  for (int k = 0; k <= m; ++k) {
    const double tk = -1.0 + 2.0 * k / m;
    double v = 1.0, d = 0.0;
    for (int j = 0; j <= m; ++j) {
      if (j == k) continue;
      const double tj = -1.0 + 2.0 * j / m;
      double prod = 1.0 / (tk - tj);
      for (int i = 0; i <= m; ++i) {
        if (i == k || i == j) continue;
        const double ti = -1.0 + 2.0 * i / m;
        prod *= (r - ti) / (tk - ti);
      }
      d += prod;
      v *= (r - tj) / (tk - tj);
    }
    l[k] = v;
    dl[k] = d;
  }
}

}  // namespace

extern "C" {

dg_status dg_implicit_init(const dg_swe_mesh* mesh, int order, int regularization, const dg_swe_params* params,
                           const dg_implicit_params* ip, dg_implicit** out) {
  if (!out) return DG_ERR_ARG;
  *out = nullptr;
  std::unique_ptr<dg_implicit> s(new dg_implicit());
  if (!mesh || !params || !ip) {
    *out = s.release();
    return ifail(*out, DG_ERR_ARG, "null argument");
  }
  if (mesh->dim != 1) {
    *out = s.release();
    return ifail(*out, DG_ERR_UNSUPPORTED, "the implicit integrator is one-dimensional");
  }
  const int m3 = ip->m3 < 0 ? order : ip->m3;
  if (!(ip->dt > 0) || ip->max_it < 1 || m3 < 0 || m3 > order || ip->linear_solver < 0 || ip->linear_solver > 1) {
    *out = s.release();
    return ifail(*out, DG_ERR_ARG, "need dt > 0, max_it >= 1, 0 <= m3 <= order, linear_solver in {0, 1}");
  }
  if (ip->n_gamma > 1 && !(ip->gamma0 > 0)) {
    *out = s.release();
    return ifail(*out, DG_ERR_ARG, "continuation needs gamma0 > 0");
  }
  if (params->flow_index != 0.0 && params->flow_index != 1.0) {
    *out = s.release();
    return ifail(*out, DG_ERR_UNSUPPORTED,
                 "the Appendix A tangent covers the Newtonian viscous part only (flow_index 1); "
                 "use dg_newton.h for the Herschel-Bulkley law");
  }
  if (ip->linear_solver == 1 && 3 * (2 * (order + 1) + m3 + 1) > 32) {
    *out = s.release();
    return ifail(*out, DG_ERR_UNSUPPORTED, "the FP32 factorization handles blocks of at most 10 unknowns (2(p+1) + m3 + 1 <= 10)");
  }
  dg_swe_ctx* c = nullptr;
  dg_status st = dg_swe_init(mesh, order, regularization, params, &c);
  if (st != DG_OK) {
    std::string m = c ? dg_swe_last_error(c) : "";
    dg_swe_destroy(c);
    *out = s.release();
    return ifail(*out, st, m);
  }
  const int64_t K = c->mesh.K;
  for (int64_t e = 0; e + 1 < K; ++e)
    if (mesh->elem_vertices[2 * e + 1] != mesh->elem_vertices[2 * (e + 1)]) {
      dg_swe_destroy(c);
      *out = s.release();
      return ifail(*out, DG_ERR_UNSUPPORTED, "1D mesh must be ordered left to right (element e+1 starts where e ends)");
    }
  s->p = order;
  s->m3 = m3;
  s->reg = regularization;
  s->K = K;
  s->prm = *params;
  s->ip = *ip;
  s->ip.m3 = m3;
  const int NP = order + 1, NE = m3 + 1;
  const RefOps& o = c->ops;
  s->wq = o.wq;
  const int NQ = o.Nq;
  s->Vq.assign(NQ * NP, 0);
  s->dVq.assign(NQ * NP, 0);
  s->VEq.assign(NQ * NE, 0);
  s->dVEq.assign(NQ * NE, 0);
  std::vector<double> l(8), dl(8);
  for (int q = 0; q < NQ; ++q) {
    lagrange1d(order, o.rq[q], l.data(), dl.data());
    for (int i = 0; i < NP; ++i) {
      s->Vq[q * NP + i] = l[i];
      s->dVq[q * NP + i] = dl[i];
    }
    lagrange1d(m3, o.rq[q], l.data(), dl.data());
    for (int i = 0; i < NE; ++i) {
      s->VEq[q * NE + i] = l[i];
      s->dVEq[q * NE + i] = dl[i];
    }
  }
  s->lf.assign(2 * NP, 0);
  s->lEf.assign(2 * NE, 0);
  for (int f = 0; f < 2; ++f) {
    lagrange1d(order, f == 0 ? -1.0 : 1.0, l.data(), dl.data());
    for (int i = 0; i < NP; ++i) s->lf[f * NP + i] = l[i];
    lagrange1d(m3, f == 0 ? -1.0 : 1.0, l.data(), dl.data());
    for (int i = 0; i < NE; ++i) s->lEf[f * NE + i] = l[i];
  }
  // reference E mass matrix inverse
  std::vector<double> ME(NE * NE, 0.0);
  for (int q = 0; q < NQ; ++q)
    for (int a = 0; a < NE; ++a)
      for (int b = 0; b < NE; ++b) ME[a * NE + b] += s->wq[q] * s->VEq[q * NE + a] * s->VEq[q * NE + b];
  s->MEinv.assign(NE * NE, 0.0);
  {  // Gauss-Jordan inverse (NE <= 4)
    std::vector<double> A(ME);
    for (int i = 0; i < NE; ++i) s->MEinv[i * NE + i] = 1.0;
    for (int k = 0; k < NE; ++k) {
      int pv = k;
      for (int r = k + 1; r < NE; ++r)
        if (std::fabs(A[r * NE + k]) > std::fabs(A[pv * NE + k])) pv = r;
      for (int j = 0; j < NE; ++j) {
        std::swap(A[k * NE + j], A[pv * NE + j]);
        std::swap(s->MEinv[k * NE + j], s->MEinv[pv * NE + j]);
      }
      const double d = 1.0 / A[k * NE + k];
      for (int j = 0; j < NE; ++j) {
        A[k * NE + j] *= d;
        s->MEinv[k * NE + j] *= d;
      }
      for (int r = 0; r < NE; ++r) {
        if (r == k) continue;
        const double f = A[r * NE + k];
        for (int j = 0; j < NE; ++j) {
          A[r * NE + j] -= f * A[k * NE + j];
          s->MEinv[r * NE + j] -= f * s->MEinv[k * NE + j];
        }
      }
    }
  }
  s->J.assign(K, 0.0);
  for (int64_t e = 0; e < K; ++e) s->J[e] = c->mesh.geo[4 * K + e];
  s->node_x.assign(c->mesh.node_xyz.begin(), c->mesh.node_xyz.end());
  if (mesh->bed) {
    s->has_bed = true;
    s->bed.assign(mesh->bed, mesh->bed + K * NP);
  }
  auto bc_of = [&](int64_t e, int f) {
    const int id = mesh->face_bc ? mesh->face_bc[e * 2 + f] : 0;
    BCEntry<double> b{};
    for (int k = 0; k < 7; ++k) {
      b.mode[k] = params->bc[id].mode[k];
      b.val[k] = params->bc[id].value[k];
    }
    return b;
  };
  s->bcL = bc_of(0, 0);
  s->bcR = bc_of(K - 1, 1);
  dg_swe_destroy(c);
  s->drv = make_idrv(*s);
  const int NB = s->nb();
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t r = off;
    off += (bytes + 255) & ~size_t(255);
    return r;
  };
  s->off.X = take(K * NB * 8);
  s->off.Uold = take(K * 2 * NP * 8);
  s->off.R = take(K * NB * 8);
  s->off.D = take(K * NB * NB * 8);
  s->off.L = take(K * NB * NB * 8);
  s->off.U = take(K * NB * NB * 8);
  s->off.Y = take(K * NB * 8);
  s->off.DX = take(K * NB * 8);
  s->off.J = take(K * 8);
  s->off.bed = take(s->has_bed ? K * NP * 8 : 0);
  s->off.red = take(64 * 8);
  s->off.st = take(sizeof(dg_implicit_stats));
  s->off.MEinv = take(NE * NE * 8);
  s->off.act = take(8);
  s->off.pt = take(K * NQ * kPt * 8);
  s->off.fc = take((K + 1) * kFc * 8);
  const size_t mixed = s->ip.linear_solver == 1 ? 1 : 0;
  s->off.Df = take(mixed * K * NB * NB * 4);
  s->off.Lf = take(mixed * K * NB * NB * 4);
  s->off.Uf = take(mixed * K * NB * NB * 4);
  s->off.bf = take(mixed * K * NB * 4);
  s->off.xf = take(mixed * K * NB * 4);
  s->off.Rr = take(mixed * K * NB * 8);
  s->ws_need = off;
  *out = s.release();
  return DG_OK;
}

size_t dg_implicit_workspace_size(const dg_implicit* s) { return s ? s->ws_need : 0; }

dg_status dg_implicit_set_stream(dg_implicit* s, void* st) {
  if (!s) return DG_ERR_ARG;
  s->stream = (cudaStream_t)st;
  return DG_OK;
}

dg_status dg_implicit_set_workspace(dg_implicit* s, void* ptr, size_t bytes) {
  if (!s) return DG_ERR_ARG;
  if (!ptr || bytes < s->ws_need) return ifail(s, DG_ERR_WORKSPACE, "workspace missing or too small");
  if (((uintptr_t)ptr & 255) != 0) return ifail(s, DG_ERR_WORKSPACE, "workspace must be 256-byte aligned");
  s->ws = (char*)ptr;
  cudaStream_t st = s->stream;
  IK(cudaMemsetAsync(s->ws, 0, s->ws_need, st));
  IK(cudaMemcpyAsync(s->ws + s->off.J, s->J.data(), s->J.size() * 8, cudaMemcpyHostToDevice, st));
  if (s->has_bed) IK(cudaMemcpyAsync(s->ws + s->off.bed, s->bed.data(), s->bed.size() * 8, cudaMemcpyHostToDevice, st));
  IK(cudaMemcpyAsync(s->ws + s->off.MEinv, s->MEinv.data(), s->MEinv.size() * 8, cudaMemcpyHostToDevice, st));
  IK(cudaStreamSynchronize(st));
  return DG_OK;
}

dg_status dg_implicit_node_coords(const dg_implicit* s, double* x) {
  if (!s || !x) return DG_ERR_ARG;
  std::memcpy(x, s->node_x.data(), s->node_x.size() * 8);
  return DG_OK;
}

dg_status dg_implicit_set_state(dg_implicit* s, const double* V, int on_device) {
  if (!s || !V) return DG_ERR_ARG;
  if (!s->ws) return ifail(s, DG_ERR_WORKSPACE, "no workspace set");
  const int NP = s->p + 1, NB = s->nb();
  const int64_t K = s->K;
  std::vector<double> hv(2 * K * NP);
  cudaStream_t st = s->stream;
  if (on_device) {
    IK(cudaMemcpyAsync(hv.data(), V, hv.size() * 8, cudaMemcpyDeviceToHost, st));
    IK(cudaStreamSynchronize(st));
  } else {
    std::memcpy(hv.data(), V, hv.size() * 8);
  }
  std::vector<double> X(K * NB, 0.0);
  for (int64_t e = 0; e < K; ++e)
    for (int i = 0; i < NP; ++i) {
      X[e * NB + i] = hv[e * NP + i];
      X[e * NB + NP + i] = hv[K * NP + e * NP + i];
    }
  IK(cudaMemcpyAsync(s->ws + s->off.X, X.data(), X.size() * 8, cudaMemcpyHostToDevice, st));
  IK(cudaMemsetAsync(s->ws + s->off.st, 0, sizeof(dg_implicit_stats), st));
  s->drv->init_E(s, st);
  IK(cudaGetLastError());
  IK(cudaStreamSynchronize(st));
  return DG_OK;
}

dg_status dg_implicit_get_state(dg_implicit* s, double* V, double* E, int on_device) {
  if (!s) return DG_ERR_ARG;
  if (!s->ws) return ifail(s, DG_ERR_WORKSPACE, "no workspace set");
  const int NP = s->p + 1, NE = s->m3 + 1, NB = s->nb();
  const int64_t K = s->K;
  std::vector<double> X(K * NB);
  IK(cudaMemcpyAsync(X.data(), s->ws + s->off.X, X.size() * 8, cudaMemcpyDeviceToHost, s->stream));
  IK(cudaStreamSynchronize(s->stream));
  std::vector<double> hv(2 * K * NP), he(K * NE);
  for (int64_t e = 0; e < K; ++e) {
    for (int i = 0; i < NP; ++i) {
      hv[e * NP + i] = X[e * NB + i];
      hv[K * NP + e * NP + i] = X[e * NB + NP + i];
    }
    for (int c = 0; c < NE; ++c) he[e * NE + c] = X[e * NB + 2 * NP + c];
  }
  const cudaMemcpyKind kind = on_device ? cudaMemcpyHostToDevice : cudaMemcpyHostToHost;
  if (V) IK(cudaMemcpy(V, hv.data(), hv.size() * 8, kind));
  if (E) IK(cudaMemcpy(E, he.data(), he.size() * 8, kind));
  return DG_OK;
}

dg_status dg_implicit_run(dg_implicit* s, int64_t n_steps, dg_implicit_stats* stats) {
  if (!s) return DG_ERR_ARG;
  if (!s->ws) return ifail(s, DG_ERR_WORKSPACE, "no workspace set");
  if (n_steps < 0) return ifail(s, DG_ERR_ARG, "n_steps < 0");
  if (n_steps > 0) s->drv->run(s, (long long)n_steps, s->stream);
  IK(cudaGetLastError());
  dg_implicit_stats h{};
  IK(cudaMemcpyAsync(&h, s->ws + s->off.st, sizeof(h), cudaMemcpyDeviceToHost, s->stream));
  IK(cudaStreamSynchronize(s->stream));
  if (stats) *stats = h;
  if (h.status != 0)
    return ifail(s, (dg_status)h.status,
                 h.status == DG_ERR_NEWTON ? "Newton did not converge within max_it" : "non-finite state");
  return DG_OK;
}

dg_status dg_implicit_active_percent(dg_implicit* s, double* pct) {
  if (!s || !pct) return DG_ERR_ARG;
  if (!s->ws) return ifail(s, DG_ERR_WORKSPACE, "no workspace set");
  s->drv->active(s, s->at<double>(s->off.act), s->stream);
  IK(cudaGetLastError());
  IK(cudaMemcpyAsync(pct, s->ws + s->off.act, 8, cudaMemcpyDeviceToHost, s->stream));
  IK(cudaStreamSynchronize(s->stream));
  return DG_OK;
}

const char* dg_implicit_last_error(const dg_implicit* s) { return s ? s->err.c_str() : "null context"; }

void dg_implicit_destroy(dg_implicit* s) { delete s; }

}  // extern "C"
