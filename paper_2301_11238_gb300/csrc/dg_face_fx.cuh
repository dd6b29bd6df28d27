// The FP64 face flux: traces interpolated in block fixed point (dg_fixed.cuh)
// and the pointwise HLL and central stress fluxes in floating point, written for
// few FP64 instructions.  Included by dg_kernels.cuh.
//
// Bound by the FP64 pipe: about 117 operations a face point in 2D (175 with
// floating-point interpolation, IEEE division and square root and FP64
// comparisons); comparisons, minima and maxima run on the integer pipe, the
// reciprocal and roots start from the FP32 unit (dg_math64.cuh).  524,288
// triangles, p = 2: 1060 -> 750 us, p = 1: 474 -> 342 us; 8,192 triangles,
// p = 2: 24.7 -> 20.6 us; 200 intervals: 10.3 -> 8.3 us.
#pragma once

namespace dgswe {

// Symmetric-gradient components the stress needs: du/dx, or (d11, d22, 2 d12).
template <int DIM>
constexpr int sym_comps() { return DIM == 1 ? 1 : 3; }

// One side of a face point: HLL ingredients and the stress row.
template <int DIM>
struct Side64 {
  double un, c;        // normal velocity, wave speed
  double U[DIM + 1];   // h, h u
  double F[DIM + 1];   // normal flux
  double m, t[DIM];    // -(Q . n)_j / 2 = m t_j
};
// nh = n / 2
template <int DIM>
__device__ __forceinline__ void side64(const double* V, const double* d, const double* n, const double* nh,
                                       const Phys<double>& ph, Side64<DIM>& s) {
  const double h = V[0];
  double un = V[1] * n[0];
  if constexpr (DIM == 2) un += V[2] * n[1];
  const double gh = ph.gc * h;
  s.un = un;
  s.c = sqrt_pos(max_pos(gh, ph.gc * ph.h_floor));
  const double q = h * un, p = h * gh;
  s.U[0] = h;
  s.F[0] = q;
#pragma unroll
  for (int j = 0; j < DIM; ++j) {
    s.U[1 + j] = h * V[1 + j];
    s.F[1 + j] = q * V[1 + j] + p * nh[j];
  }
  if constexpr (DIM == 1) {
    s.m = (stress_mu1<double>(d[0], ph) * h) * (-0.5 * ph.rho_inv);
    s.t[0] = (2.0 * d[0]) * n[0];
  } else {
    const double tr = d[0] + d[1], e = 0.5 * d[2];
    const double s2 = 0.5 * (d[0] * d[0] + d[1] * d[1] + tr * tr + d[2] * e);
    s.m = (stress_mu2<double>(s2, ph) * h) * (-0.5 * ph.rho_inv);
    s.t[0] = (d[0] + tr) * n[0] + e * n[1];
    s.t[1] = e * n[0] + (d[1] + tr) * n[1];
  }
}

// Weighted numerical flux of one point: HLL for F minus the central flux of Q.
template <int DIM>
__device__ __forceinline__ void flux64(const double* Vm, const double* Vp, const double* dm, const double* dp,
                                       const double* n, const Phys<double>& ph, double w, double* out) {
  double nh[DIM];
#pragma unroll
  for (int j = 0; j < DIM; ++j) nh[j] = 0.5 * n[j];
  Side64<DIM> a, b;
  side64<DIM>(Vm, dm, n, nh, ph, a);
  side64<DIM>(Vp, dp, n, nh, ph, b);
  const double SL = min_f64(a.un - a.c, b.un - b.c), SR = max_f64(a.un + a.c, b.un + b.c);
  double Fn[DIM + 1];
  if (__double2hiint(SL) >= 0) {
#pragma unroll
    for (int v = 0; v < DIM + 1; ++v) Fn[v] = a.F[v];
  } else if (__double2hiint(SR) < 0) {
#pragma unroll
    for (int v = 0; v < DIM + 1; ++v) Fn[v] = b.F[v];
  } else {
    const double inv = rcp_pos(SR - SL);
    const double x = SR * inv, y = -SL * inv, z = SL * x;
#pragma unroll
    for (int v = 0; v < DIM + 1; ++v) Fn[v] = x * a.F[v] + (y * b.F[v] + z * (b.U[v] - a.U[v]));
  }
  out[0] = w * Fn[0];
#pragma unroll
  for (int j = 0; j < DIM; ++j) out[1 + j] = w * (Fn[1 + j] + (a.m * a.t[j] + b.m * b.t[j]));
}

// Traces of one side of a face at its nodes, as operands with one exponent per
// field: h, u, then the symmetric-gradient components.
template <int DIM, int P>
struct Trace64 {
  static constexpr int NX = DIM + 1 + sym_comps<DIM>();
  Fx x[NX][Sh<DIM, P>::NFP];
  int e[NX];  // exponent of the unit: results of a table with scale cs are r 2^(e - cs)
};
template <int DIM, int P, bool COH>
__device__ __forceinline__ void load_trace64(const double* __restrict__ V, const double* __restrict__ E, size_t KN,
                                             size_t eo, const int8_t* fm, bool flip, Trace64<DIM, P>& t) {
  using S = Sh<DIM, P>;
  constexpr int NFP = S::NFP, NV = S::NV;
  size_t at[NFP];
#pragma unroll
  for (int k = 0; k < NFP; ++k) at[k] = eo + fm[flip ? NFP - 1 - k : k];
#pragma unroll
  for (int v = 0; v < NV + 2; ++v) {  // h, u, d11, d22
    const double* src = v < NV ? V + v * KN : E + (v == NV ? 0 : 3) * KN;
    double x[NFP];
    int e = 0;
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      x[k] = DG_LDC(COH, src, at[k]);
      e = max(e, fx_exp(x[k]));
    }
#pragma unroll
    for (int k = 0; k < NFP; ++k) t.x[v][k] = fx_from<5>(x[k], e);
    t.e[v] = e - 1024;
  }
  {  // 2 d12 = E_12 + E_21
    double x[NFP], y[NFP];
    int e = 0;
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      x[k] = DG_LDC(COH, E, KN + at[k]);
      y[k] = DG_LDC(COH, E, 2 * KN + at[k]);
      e = max(e, max(fx_exp(x[k]), fx_exp(y[k])));
    }
#pragma unroll
    for (int k = 0; k < NFP; ++k) {
      const Fx p = fx_from<4>(x[k], e), q = fx_from<4>(y[k], e);
      t.x[NV + 2][k] = Fx{p.h + q.h, p.l + q.l};
    }
    t.e[NV + 2] = e - 1023;
  }
}
template <int DIM, int P>
__device__ __forceinline__ void trace_at(const Trace64<DIM, P>& t, const FaceOps<DIM, P, double>& ops, int m,
                                         double* V, double* d) {
  using S = Sh<DIM, P>;
  constexpr int NFP = S::NFP, NV = S::NV;
#pragma unroll
  for (int v = 0; v < Trace64<DIM, P>::NX; ++v) {
    FxAcc s{0, 0};
#pragma unroll
    for (int k = 0; k < NFP; ++k) fx_mac(s, t.x[v][k], ops.Lfx[m * NFP + k]);
    const double r = fx_to(fx_sum(s), fx_scale(t.e[v] - ops.cs, t.e[v] <= kFxMaxExp - 1024));
    if (v < NV) V[v] = r;
    else d[v - NV] = r;
  }
}

// Face fc: its points m0 .. m1 - 1 (all of them, or one).
template <int DIM, int P, bool COH>
__device__ __forceinline__ void face_fx(int fc, int m0, int m1, int e1, int f1, int e2, int f2, const double (&n)[DIM],
                                        double wsj, int K, int F, const double* __restrict__ V,
                                        const double* __restrict__ E, double* __restrict__ wflux,
                                        const FaceOps<DIM, P, double>& ops, const Phys<double>& ph,
                                        const BCEntry<double>* __restrict__ bct) {
  using S = Sh<DIM, P>;
  constexpr int NP = S::NP, NFP = S::NFP, NFQ = S::NFQ, NV = S::NV, ND = sym_comps<DIM>();
  const size_t KN = (size_t)K * NP, FQ = (size_t)F * NFQ;
  const bool interior = e2 >= 0;
  if constexpr (DIM == 1) {
    // one node, one point: no interpolation
    double Vm[NV], Vp[NV], dm[ND], dp[ND], out[NV];
    const size_t a = (size_t)e1 * NP + ops.fmask[f1], b = interior ? (size_t)e2 * NP + ops.fmask[f2] : a;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      Vm[v] = DG_LDC(COH, V, v * KN + a);
      Vp[v] = DG_LDC(COH, V, v * KN + b);
    }
    dm[0] = DG_LDC(COH, E, a);
    dp[0] = DG_LDC(COH, E, b);
    if (!interior) {
      const BCEntry<double> bc = bct[-1 - e2];
      ghost_V<DIM, double>(Vm, n, bc, Vp);
      ghost_E<DIM, double>(dm, bc, dp);
    }
    flux64<DIM>(Vm, Vp, dm, dp, n, ph, ops.wf[0] * wsj, out);
#pragma unroll
    for (int v = 0; v < NV; ++v) wflux[v * FQ + fc] = out[v];
  } else {
    Trace64<DIM, P> tm, tp;
    load_trace64<DIM, P, COH>(V, E, KN, (size_t)e1 * NP, ops.fmask + f1 * NFP, false, tm);
    if (interior) load_trace64<DIM, P, COH>(V, E, KN, (size_t)e2 * NP, ops.fmask + f2 * NFP, true, tp);
#pragma unroll 1
    for (int m = m0; m < m1; ++m) {
      double Vm[NV], Vp[NV], dm[ND], dp[ND], out[NV];
      trace_at<DIM, P>(tm, ops, m, Vm, dm);
      if (interior) {
        trace_at<DIM, P>(tp, ops, m, Vp, dp);
      } else {
        const BCEntry<double> bc = bct[-1 - e2];
        ghost_V<DIM, double>(Vm, n, bc, Vp);
        dp[0] = bc.mode[3] == 1 ? bc.val[3] : dm[0];
        dp[1] = bc.mode[6] == 1 ? bc.val[6] : dm[1];
        dp[2] = dm[2];
        if (bc.mode[4] == 1 || bc.mode[5] == 1) {
          // a prescribed E_12 or E_21: the two components apart
          double x = 0.0, y = 0.0;
          for (int k = 0; k < NFP; ++k) {
            const size_t a = (size_t)e1 * NP + ops.fmask[f1 * NFP + k];
            x += ops.Lf[m * NFP + k] * DG_LDC(COH, E, KN + a);
            y += ops.Lf[m * NFP + k] * DG_LDC(COH, E, 2 * KN + a);
          }
          dp[2] = (bc.mode[4] == 1 ? bc.val[4] : x) + (bc.mode[5] == 1 ? bc.val[5] : y);
        }
      }
      flux64<DIM>(Vm, Vp, dm, dp, n, ph, ops.wf[m] * wsj, out);
#pragma unroll
      for (int v = 0; v < NV; ++v) wflux[v * FQ + (size_t)fc * NFQ + m] = out[v];
    }
  }
}

}  // namespace dgswe
